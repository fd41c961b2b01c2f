// Eddy currents of a conducting magnet (Sec. III.B, the Torres method): the
// cell kernels of the electric-potential step and of the current.
//
// E_sol (step 1) and H_eddy (step 4) are cross products with the kernel S of
// the scalar potential, sum_j V(r_j) x S(r_i - r_j); each component of such a
// product is a dot product of S with a rearranged field,
//   (V x S)_x = S . (0, -V_z, V_y),  (V x S)_y = S . (V_z, 0, -V_x),
//   (V x S)_z = S . (-V_y, V_x, 0),
// so the host runs the potential path three times (k_cross_input builds the
// inputs, k_scale_into collects the outputs).
//
// Step 2, Laplace's equation for phi_E in the magnet with d phi / dn = E_sol . n
// on its surface, cell-centred: in every cell the sum over axes of
// w_a sum_{neighbours present} (phi_nb - phi) equals b = the surface fluxes,
// w_a = 1 / d_a^2, b = -sum_{a: + face on the surface} E_sol,a / d_a
// + sum_{a: - face on the surface} E_sol,a / d_a, with the mean of b removed
// (compatibility).  Solved by red-black successive over-relaxation in FP64
// (phi stored in FP32 would leave a residual floor of ~n 2e-7 of the source,
// too coarse to certify convergence); the host checks the residual every few
// sweeps, bounds the number of sweeps, and removes the mean of phi at the end.
#include <cuda_runtime.h>

#include "mm_internal.h"

namespace mm {

struct CellIdx {
  int x, y, z;
};

__device__ __forceinline__ CellIdx cell_of(size_t i, int nx, int ny) {
  const unsigned nxy = (unsigned)nx * (unsigned)ny;
  const int z = (int)((unsigned)i / nxy);
  const unsigned rem = (unsigned)i - (unsigned)z * nxy;
  const int y = (int)(rem / (unsigned)nx);
  return CellIdx{(int)(rem - (unsigned)y * (unsigned)nx), y, z};
}

__global__ void __launch_bounds__(256) k_cross_input(const float* __restrict__ V, size_t N, int comp,
                                                     float* __restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float vx = V[i], vy = V[N + i], vz = V[2 * N + i];
  float a = 0.f, b = 0.f, c = 0.f;
  if (comp == 0) { b = -vz; c = vy; }
  else if (comp == 1) { a = vz; c = -vx; }
  else { a = -vy; b = vx; }
  out[i] = a; out[N + i] = b; out[2 * N + i] = c;
}

__global__ void __launch_bounds__(256) k_scale_into(const float* __restrict__ in, size_t N, float s,
                                                    float* __restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) out[i] = s * in[i];
}

__global__ void __launch_bounds__(256) k_accumulate(const float* __restrict__ in, size_t N,
                                                    float* __restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) out[i] += in[i];
}

// b of every cell and per-block sums of b (for its mean)
__global__ void __launch_bounds__(256) k_eddy_source(const float* __restrict__ E, int nx, int ny, int nz,
                                                     double idx_, double idy, double idz, double* __restrict__ b,
                                                     double* __restrict__ part) {
  __shared__ double red[256];
  const size_t N = (size_t)nx * ny * nz;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (i < N) {
    const CellIdx c = cell_of(i, nx, ny);
    const double ex = E[i], ey = E[N + i], ez = E[2 * N + i];
    if (c.x == nx - 1) v -= ex * idx_;
    if (c.x == 0) v += ex * idx_;
    if (c.y == ny - 1) v -= ey * idy;
    if (c.y == 0) v += ey * idy;
    if (c.z == nz - 1) v -= ez * idz;
    if (c.z == 0) v += ez * idz;
    b[i] = v;
  }
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// fixed-order sum of nparts doubles into *out (one block)
__global__ void __launch_bounds__(256) k_sum_parts(const double* __restrict__ part, int nparts, double scale,
                                                   double* __restrict__ out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int k = threadIdx.x; k < nparts; k += blockDim.x) s += part[k];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int t = 128; t > 0; t >>= 1) {
    if (threadIdx.x < t) red[threadIdx.x] += red[threadIdx.x + t];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = scale * red[0];
}

// the source with its mean removed, in place
__global__ void __launch_bounds__(256) k_sub_mean(double* __restrict__ b, size_t N, const double* __restrict__ mean) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) b[i] -= *mean;
}

// Weights of the SOR update: w per axis, and c = omega / (sum of the weights of
// the neighbours present), by the number of neighbours along each axis.
struct SorCoef {
  double wx, wy, wz, omega1;  // omega1 = 1 - omega
  double c[27];               // [present x + 3 present y + 9 present z]
};

// One colour of a red-black SOR sweep, cells with (x + y + z) % 2 == colour, a
// thread per cell of the colour: phi <- (1 - omega) phi + c (sum w phi_nb - b').
// The FP64 pipe is what bounds it (two operations per clock and SM): nine
// operations a cell, no division (the sum, the weights and the quotient written
// out per neighbour were about 35: 18 us a colour at 64^3, now 6 us).
__global__ void __launch_bounds__(256) k_sor(double* __restrict__ phi, const double* __restrict__ b, int nx, int ny,
                                             int nz, const SorCoef C, int colour) {
  const unsigned nh = (unsigned)(nx + 1) >> 1;  // cells of a colour per row, at most
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned row = i / nh;
  pdl_wait();
  if (row >= (unsigned)ny * (unsigned)nz) return;
  const int z = (int)(row / (unsigned)ny), y = (int)(row - (unsigned)z * (unsigned)ny);
  const int x = 2 * (int)(i - row * nh) + ((y + z + colour) & 1);
  if (x >= nx) return;
  const size_t p = (size_t)row * nx + x, sz = (size_t)nx * ny;
  const bool xm = x > 0, xp = x < nx - 1, ym = y > 0, yp = y < ny - 1, zm = z > 0, zp = z < nz - 1;
  const int present = (xm + xp) + 3 * (ym + yp) + 9 * (zm + zp);
  if (present == 0) return;  // a single cell: phi = 0
  const double sx = (xm ? phi[p - 1] : 0.0) + (xp ? phi[p + 1] : 0.0);
  const double sy = (ym ? phi[p - nx] : 0.0) + (yp ? phi[p + nx] : 0.0);
  const double s_z = (zm ? phi[p - sz] : 0.0) + (zp ? phi[p + sz] : 0.0);
  const double t = fma(C.wx, sx, fma(C.wy, sy, fma(C.wz, s_z, -b[p])));
  phi[p] = fma(C.c[present], t, C.omega1 * phi[p]);
}

// Non-negative doubles compare like their bit patterns (the integer pipe, not
// the FP64 one); a NaN counts as zero, as fmax has it.
__device__ __forceinline__ unsigned long long max_bits(double v) {
  return v > 0.0 ? (unsigned long long)__double_as_longlong(v) : 0ull;
}
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

// block maxima of r and bb and the block sum of p, in thread 0, in a fixed order
__device__ __forceinline__ void residual_reduce(unsigned long long& r, unsigned long long& bb, double& p) {
  __shared__ unsigned long long rs[8], bs[8];
  __shared__ double ps[8];
  for (int o = 16; o > 0; o >>= 1) {
    r = umax64(r, __shfl_down_sync(0xffffffffu, r, o));
    bb = umax64(bb, __shfl_down_sync(0xffffffffu, bb, o));
    p += __shfl_down_sync(0xffffffffu, p, o);
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    rs[w] = r; bs[w] = bb; ps[w] = p;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 1; k < 8; ++k) {
      r = umax64(r, rs[k]);
      bb = umax64(bb, bs[k]);
      p += ps[k];
    }
}

// per-block max |A phi - b'| and max |b'|, and the block sum of phi (its mean)
__global__ void __launch_bounds__(256) k_sor_residual(const double* __restrict__ phi, const double* __restrict__ b,
                                                      int nx, int ny, int nz, double wx, double wy, double wz,
                                                      double* __restrict__ part) {
  const size_t N = (size_t)nx * ny * nz;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  double r = 0.0, bb = 0.0, p = 0.0;
  if (i < N) {
    const CellIdx c = cell_of(i, nx, ny);
    const double f = phi[i];
    double s = 0.0;
    if (c.x > 0) s += wx * (phi[i - 1] - f);
    if (c.x < nx - 1) s += wx * (phi[i + 1] - f);
    if (c.y > 0) s += wy * (phi[i - nx] - f);
    if (c.y < ny - 1) s += wy * (phi[i + nx] - f);
    if (c.z > 0) s += wz * (phi[i - (size_t)nx * ny] - f);
    if (c.z < nz - 1) s += wz * (phi[i + (size_t)nx * ny] - f);
    r = fabs(s - b[i]);
    bb = fabs(b[i]);
    p = f;
  }
  unsigned long long rb = max_bits(r), bbb = max_bits(bb);
  residual_reduce(rb, bbb, p);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = __longlong_as_double((long long)rb);
    part[3 * blockIdx.x + 1] = __longlong_as_double((long long)bbb);
    part[3 * blockIdx.x + 2] = p;
  }
}

// out[0] = max residual, out[1] = max |b'|, out[2] = mean phi (one block)
__global__ void __launch_bounds__(256) k_residual_reduce(const double* __restrict__ part, int nparts, double invN,
                                                         double* __restrict__ out) {
  unsigned long long r = 0ull, bb = 0ull;
  double p = 0.0;
  for (int k = threadIdx.x; k < nparts; k += blockDim.x) {
    r = umax64(r, max_bits(part[3 * k]));
    bb = umax64(bb, max_bits(part[3 * k + 1]));
    p += part[3 * k + 2];
  }
  residual_reduce(r, bb, p);
  if (threadIdx.x == 0) {
    out[0] = __longlong_as_double((long long)r);
    out[1] = __longlong_as_double((long long)bb);
    out[2] = p * invN;
  }
}

// E_irrot = -grad (phi - mean phi) with the boundary condition's ghost values,
// J = sigma (E_sol + E_irrot)
__global__ void __launch_bounds__(256) k_eddy_current(const double* __restrict__ phi, const double* __restrict__ stats,
                                                      const float* __restrict__ E, int nx, int ny, int nz, double dx,
                                                      double dy, double dz, double sigma, float* __restrict__ J) {
  const size_t N = (size_t)nx * ny * nz;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const CellIdx c = cell_of(i, nx, ny);
  const double mean = stats[2];
  const double f = phi[i] - mean;
  const double ex = E[i], ey = E[N + i], ez = E[2 * N + i];
  const double xp = c.x < nx - 1 ? phi[i + 1] - mean : f + dx * ex;
  const double xm = c.x > 0 ? phi[i - 1] - mean : f - dx * ex;
  const double yp = c.y < ny - 1 ? phi[i + nx] - mean : f + dy * ey;
  const double ym = c.y > 0 ? phi[i - nx] - mean : f - dy * ey;
  const size_t sz = (size_t)nx * ny;
  const double zp = c.z < nz - 1 ? phi[i + sz] - mean : f + dz * ez;
  const double zm = c.z > 0 ? phi[i - sz] - mean : f - dz * ez;
  J[i] = (float)(sigma * (ex - (xp - xm) / (2.0 * dx)));
  J[N + i] = (float)(sigma * (ey - (yp - ym) / (2.0 * dy)));
  J[2 * N + i] = (float)(sigma * (ez - (zp - zm) / (2.0 * dz)));
}

// Coupling into the time step: B = mu0 (H_demag + H_stray + H_ext + Ms y) of
// the step's last evaluation; with a previous B, dB/dt = (B - B_prev) / dt;
// then B_prev = B.
__global__ void __launch_bounds__(256) k_flux_rate(const float* __restrict__ Hself, const float* __restrict__ Hstray,
                                                   const float* __restrict__ y, size_t N, float hx, float hy, float hz,
                                                   float Ms, float mu0, float inv_dt, int have_prev,
                                                   float* __restrict__ Bprev, float* __restrict__ Bdot) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float he[3] = {hx, hy, hz};
  for (int c = 0; c < 3; ++c) {
    const size_t k = c * N + i;
    const float B = mu0 * (Hself[k] + Hstray[k] + he[c] + Ms * y[k]);
    if (have_prev) Bdot[k] = (B - Bprev[k]) * inv_dt;
    Bprev[k] = B;
  }
}

static unsigned blocks(size_t N) { return (unsigned)((N + 255) / 256); }

cudaError_t launch_flux_rate(const float* Hself, const float* Hstray, const float* y, size_t N, const double hext[3],
                             double Ms, double dt, int have_prev, float* Bprev, float* Bdot, cudaStream_t st) {
  k_flux_rate<<<blocks(N), 256, 0, st>>>(Hself, Hstray, y, N, (float)hext[0], (float)hext[1], (float)hext[2],
                                         (float)Ms, (float)(4e-7 * 3.14159265358979323846), (float)(1.0 / dt),
                                         have_prev, Bprev, Bdot);
  return cudaGetLastError();
}

cudaError_t launch_cross_input(const float* V, size_t N, int comp, float* out, cudaStream_t st) {
  k_cross_input<<<blocks(N), 256, 0, st>>>(V, N, comp, out);
  return cudaGetLastError();
}

cudaError_t launch_scale_into(const float* in, size_t N, float s, float* out, cudaStream_t st) {
  k_scale_into<<<blocks(N), 256, 0, st>>>(in, N, s, out);
  return cudaGetLastError();
}

cudaError_t launch_accumulate(const float* in, size_t N, float* out, cudaStream_t st) {
  if (N == 0) return cudaSuccess;
  k_accumulate<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(in, N, out);
  return cudaGetLastError();
}

int eddy_blocks(size_t N) { return (int)blocks(N); }

cudaError_t launch_eddy_source(const float* E, int nx, int ny, int nz, const double d[3], double* b, double* part,
                               double* bmean, cudaStream_t st) {
  const size_t N = (size_t)nx * ny * nz;
  k_eddy_source<<<blocks(N), 256, 0, st>>>(E, nx, ny, nz, 1.0 / d[0], 1.0 / d[1], 1.0 / d[2], b, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sum_parts<<<1, 256, 0, st>>>(part, (int)blocks(N), 1.0 / (double)N, bmean);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sub_mean<<<blocks(N), 256, 0, st>>>(b, N, bmean);
  return cudaGetLastError();
}

cudaError_t launch_sor_sweeps(double* phi, const double* b, int nx, int ny, int nz, const double d[3], double omega,
                              int sweeps, cudaStream_t st) {
  SorCoef C;
  C.wx = 1.0 / (d[0] * d[0]); C.wy = 1.0 / (d[1] * d[1]); C.wz = 1.0 / (d[2] * d[2]);
  C.omega1 = 1.0 - omega;
  for (int k = 0; k < 27; ++k) {
    const double w = (k % 3) * C.wx + (k / 3 % 3) * C.wy + (k / 9) * C.wz;
    C.c[k] = w > 0.0 ? omega / w : 0.0;
  }
  const size_t n = (size_t)((nx + 1) / 2) * ny * nz;
  for (int k = 0; k < sweeps; ++k)
    for (int colour = 0; colour < 2; ++colour) {
      cudaError_t e = launch_chained(k_sor, blocks(n), 256, 0, st, phi, b, nx, ny, nz, C, colour);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

cudaError_t launch_sor_residual(const double* phi, const double* b, int nx, int ny, int nz, const double d[3],
                                double* part, double* stats, cudaStream_t st) {
  const size_t N = (size_t)nx * ny * nz;
  const double wx = 1.0 / (d[0] * d[0]), wy = 1.0 / (d[1] * d[1]), wz = 1.0 / (d[2] * d[2]);
  k_sor_residual<<<blocks(N), 256, 0, st>>>(phi, b, nx, ny, nz, wx, wy, wz, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_residual_reduce<<<1, 256, 0, st>>>(part, (int)blocks(N), 1.0 / (double)N, stats);
  return cudaGetLastError();
}

cudaError_t launch_eddy_current(const double* phi, const double* stats, const float* E, int nx, int ny, int nz,
                                const double d[3], double sigma, float* J, cudaStream_t st) {
  const size_t N = (size_t)nx * ny * nz;
  k_eddy_current<<<blocks(N), 256, 0, st>>>(phi, stats, E, nx, ny, nz, d[0], d[1], d[2], sigma, J);
  return cudaGetLastError();
}

}  // namespace mm
