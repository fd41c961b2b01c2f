// FFT passes for thick magnets (nz > 4): the convolution of Sec. III.A with z
// by FFT, on a Qx x Qy x Qz circular grid.
//
//   x pass (k_xfwd, shared with thin films)          -> X1[plane][kx][y]
//   y forward (k_yfwd3): y FFT of each column        -> Y3[kx][ypos][plane]
//   z pass (k_zpass3): per (kx, y position) the z FFT of the three components,
//       H = -N.M and phi = S.M against the 3D kernel spectra, the inverse z
//       FFT, and the z prefilter of phi on the box  -> Z[plane][kx][ypos]
//   or, for sources of up to kMaxNzDirect layers, the direct z sum (k_zmix3)
//       with thin-film spectra (z prefilter folded in), y in natural order
//   y inverse (k_yinv3): inverse y FFT, demag rows and y prefilter
//                                                    -> Y[plane][kx][row]
//   x pass (k_xinv, shared)                          -> real rows
//
// Planes are (component, z layer) = c nz + z.  Y3 keeps the planes of one
// (kx, y position) contiguous so the z pass reads them as whole runs, and Z
// keeps y positions contiguous for the y inverse.  y positions stay in the
// DIF order of the forward transform; the inverse (DIT) takes them back.
//
// Kernel spectra (FP32, generated once in FP64) are stored for kx <= Qx/2,
// ky <= Qy/2, kz <= Qz/2.  Every component of N and S has a parity in each
// axis: the six N spectra are real (each off-diagonal is odd in exactly two
// axes), the three S spectra imaginary (each odd in one); mirrored ky or kz
// flips the sign of the components odd in that axis.
#include <algorithm>

#include "fft.cuh"
#include "fft2.cuh"
#include "mm_internal.h"
#include "prefilter.cuh"
#include "umma.cuh"

namespace mm {

// this translation unit's copy of the small-DFT roots (see fft.cuh)
cudaError_t init_fft_constants_3d() { return upload_roots(); }

// The block's lines from memory: f(l, i) loads point i < n of line l < nl, and
// sm[l ldl + i] takes it, kLineBatch loads of a thread in flight (one at a time,
// a short line waited out the memory latency once per line).
constexpr int kLineBatch = 8;
template <typename Ld>
__device__ __forceinline__ void load_lines(float2* sm, int ldl, int nl, int n, Ld f) {
  // a warp takes 32 consecutive points of a line at a time
  const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per = (n + 31) >> 5, runs = nl * per;
  for (int r0 = warp; r0 < runs; r0 += kLineBatch * warps) {
    float2 v[kLineBatch];
    int l = r0 / per, c = r0 - l * per;  // line and run of the line, walked without divisions
    const int l0 = l, c0 = c;
#pragma unroll
    for (int u = 0; u < kLineBatch; ++u) {
      const int i = (c << 5) + lane;
      if (l < nl && i < n) v[u] = f(l, i);
      c += warps;
      while (c >= per) { c -= per; ++l; }
    }
    l = l0;
    c = c0;
#pragma unroll
    for (int u = 0; u < kLineBatch; ++u) {
      const int i = (c << 5) + lane;
      if (l < nl && i < n) sm[l * ldl + i] = v[u];
      c += warps;
      while (c >= per) { c -= per; ++l; }
    }
  }
}

// ------------------------------------------------------------------ y forward
// FIXP > 0: every job's y plan is fixed plan FIXP, run with its lengths as constants.
template <unsigned RSET, int FIXP>
__global__ void __launch_bounds__(256, 3) k_yfwd3(const Launch<YFwdJob> Lc) {
  extern __shared__ float2 sm[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const YFwdJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int ng = (J.planes + J.group - 1) / J.group;
  const int kx = tile / ng;
  const int p0 = (tile - kx * ng) * J.group;
  const int np = min(J.group, J.planes - p0);
  const int Q = FIXP ? FixedPlan<FIXP ? FIXP : 1>::L : J.fy.plan.L;
  const int ldl = Q + 1;  // odd stride: the plane-fastest reads below spread over the banks
  const int ny = J.ny;
  const float2* in0 = J.in + ((size_t)p0 * J.kxh + kx) * ny;
  const size_t pstride = (size_t)J.kxh * ny;
  load_lines(sm, ldl, np, ny, [&](int l, int y) { return in0[l * pstride + y]; });
  __syncthreads();
  // rows [ny, Q) are zero padding: the first stage takes them as zero unread
  if constexpr (FIXP > 0)
    fft_smem_plan<kFwdDif, FIXP, FixedPlan<FIXP>::L + 1>(sm, np, J.fy.plan, J.fy.tw_f, 0, blockDim.x, ny);
  else
    fft_smem<kFwdDif, float2, RSET>(sm, ldl, np, J.fy.plan, J.fy.tw_f, 0, blockDim.x, ny);
  if (J.natural) {
    // frequency ky read from its DIF position: whole contiguous output rows
    for (int l = 0; l < np; ++l) {
      float2* row = J.out + ((size_t)(p0 + l) * J.kxh + kx) * Q;
      for (int k = threadIdx.x; k < Q; k += blockDim.x) row[k] = sm[l * ldl + __ldg(J.fy.pos + k)];
    }
    return;
  }
  float2* dst = J.out + (size_t)kx * Q * J.planes + p0;
  if (np == 16) {
    for (int i = threadIdx.x; i < 16 * Q; i += blockDim.x) dst[(size_t)(i >> 4) * J.planes + (i & 15)] = sm[(i & 15) * ldl + (i >> 4)];
    return;
  }
  for (int i = threadIdx.x; i < Q * np; i += blockDim.x) {
    const int p = i / np, l = i - p * np;
    dst[(size_t)p * J.planes + l] = sm[l * ldl + p];
  }
}

// ------------------------------------------------------------------ z pass
__device__ __forceinline__ float2 c_i_times(float2 m) { return make_float2(-m.y, m.x); }

template <unsigned RSET>
__global__ void __launch_bounds__(256, 2) k_zpass3(const Launch<ZJob> Lc) {
  extern __shared__ float2 sm[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const ZJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int Qy = J.fy.plan.L, Qz = J.fz.plan.L;
  const int zt = J.ztile;
  const int zl = 31 - __clz(zt);  // zt is a power of two
  const int npt = (Qy + zt - 1) >> zl;
  const int kx = tile / npt;
  const int y0 = (tile - kx * npt) << zl;
  const int nt = min(zt, Qy - y0);
  const int nz = J.nz, P3 = 3 * nz;
  const int ldz = Qz + 1;
  // lines: t * 3 + c (input, then H in place) for t < nt; phi line t at 3 zt + t
  float2* phi = sm + 3 * zt * ldz;
  int* tab = reinterpret_cast<int*>(sm + 4 * zt * ldz);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;

  // the 3 nz values of a y position are one run in memory, nz of each component
  const float2* src = J.in + ((size_t)kx * Qy + y0) * P3;
  load_lines(sm, ldz, 3 * nt, nz, [&](int l, int z) { return src[(size_t)l * nz + z]; });
  if (J.do_C) build_pref_table(tab, J.r + 2 * kPrefWarm + kZChunk, J.box_lo, J.box_len, J.start, Qz, nullptr);
  __syncthreads();
  // layers [nz, Qz) are zero padding: the first stage takes them as zero unread
  fft_smem<kFwdDif, float2, RSET>(sm, ldz, 3 * nt, J.fz.plan, J.fz.tw_f, 0, blockDim.x, nz);

  // spectral products at the pair (kz, Qz - kz): a warp per y position, its
  // lanes along kz, the kernel values of the next 32 kz on their way meanwhile
  const int half = Qz >> 1;
  const size_t kstride = (size_t)J.kxh * J.kyq * J.kzq;
  for (int t = warp; t < nt; t += warps) {
    const int ky = __ldg(J.fy.freq + y0 + t);
    const bool ym = 2 * ky > Qy;
    const float sy = ym ? -1.f : 1.f;
    const size_t krow = ((size_t)kx * J.kyq + (ym ? Qy - ky : ky)) * J.kzq;
    float2* line = sm + 3 * t * ldz;
    for (int kz = lane; kz <= half; kz += 32) {
      const bool two = kz != 0 && 2 * kz != Qz;
      const int q0 = __ldg(J.fz.pos + kz);
      const int q1 = two ? __ldg(J.fz.pos + Qz - kz) : q0;
      float nv[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, sv[3] = {0.f, 0.f, 0.f};
      if (J.do_H)
#pragma unroll
        for (int c = 0; c < 6; ++c) nv[c] = __ldg(J.N3 + c * kstride + krow + kz);
      if (J.do_C)
#pragma unroll
        for (int c = 0; c < 3; ++c) sv[c] = __ldg(J.S3 + c * kstride + krow + kz);
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 1 && !two) break;
        const int q = side ? q1 : q0;
        const float sz = side ? -1.f : 1.f;
        const float2 mx = line[q], my = line[ldz + q], mz = line[2 * ldz + q];
        if (J.do_C) {
          // phi = i (Sx mx + Sy my + Sz mz); Sy odd in y, Sz odd in z
          const float ax = sv[0], ay = sy * sv[1], az = sz * sv[2];
          phi[t * ldz + q] = c_i_times(make_float2(ax * mx.x + ay * my.x + az * mz.x,
                                                   ax * mx.y + ay * my.y + az * mz.y));
        }
        if (J.do_H) {
          // N real: xy odd in y, xz odd in z, yz odd in both
          const float nxx = nv[0], nyy = nv[1], nzz = nv[2];
          const float nxy = sy * nv[3], nxz = sz * nv[4], nyz = sy * sz * nv[5];
          line[q] = make_float2(nxx * mx.x + nxy * my.x + nxz * mz.x, nxx * mx.y + nxy * my.y + nxz * mz.y);
          line[ldz + q] = make_float2(nxy * mx.x + nyy * my.x + nyz * mz.x, nxy * mx.y + nyy * my.y + nyz * mz.y);
          line[2 * ldz + q] = make_float2(nxz * mx.x + nyz * my.x + nzz * mz.x, nxz * mx.y + nyz * my.y + nzz * mz.y);
        }
      }
    }
  }
  __syncthreads();
  if (J.do_H) fft_smem<kInvDit, float2, RSET>(sm, ldz, 3 * nt, J.fz.plan, J.fz.tw_f, 0, blockDim.x);
  if (J.do_C) fft_smem<kInvDit, float2, RSET>(phi, ldz, nt, J.fz.plan, J.fz.tw_f, 0, blockDim.x);

  // outputs with the y position fastest: runs of the tile's positions
  if (J.do_H) {
    for (int c = 0; c < 3; ++c) {
      float2* out = J.outH + ((size_t)c * nz * J.kxh + kx) * Qy + y0;
      for (int i = threadIdx.x; i < nz << zl; i += blockDim.x) {
        const int z = i >> zl, t = i & (zt - 1);
        if (t < nt) out[(size_t)z * J.kxh * Qy + t] = sm[(t * 3 + c) * ldz + z];
      }
    }
  }
  if (J.do_C) {
    const int r = J.r;
    float2* out = J.outC + (size_t)kx * Qy + y0;
    const size_t ostride = (size_t)J.kxh * Qy;
    if (J.fir) {
      const int nch = (r + kZChunk - 1) / kZChunk;
      for (int i = threadIdx.x; i < nch << zl; i += blockDim.x) {
        const int t = i & (zt - 1);
        const int k0 = (i >> zl) * kZChunk;
        if (t >= nt) continue;
        const float2* line = phi + t * ldz;
        prefilter_chunk<kZChunk, f2>(
            k0, r, [&](int jj) { return f2(line[tab[jj]]); },
            [&](int k, f2 v) { out[k * ostride + t] = make_float2(v.x, v.y); });
      }
    } else {
      for (int i = threadIdx.x; i < r << zl; i += blockDim.x) {
        const int k = i >> zl, t = i & (zt - 1);
        if (t < nt) out[k * ostride + t] = phi[t * ldz + tab[k + kPrefWarm]];
      }
    }
  }
}

// ------------------------------------------------------------------ y inverse
template <unsigned RSET, int FIXP>
__global__ void __launch_bounds__(256, 3) k_yinv3(const Launch<YInvJob> Lc) {
  extern __shared__ float2 sm[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const YInvJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int ng = (J.planes + J.group - 1) / J.group;
  const int kx = tile / ng;
  const int p0 = (tile - kx * ng) * J.group;
  const int np = min(J.group, J.planes - p0);
  const int Q = FIXP ? FixedPlan<FIXP ? FIXP : 1>::L : J.fy.plan.L;
  const int ldl = Q + 1;
  int* tab = reinterpret_cast<int*>(sm + J.group * ldl);
  const float2* in0 = J.in + ((size_t)p0 * J.kxh + kx) * Q;
  const size_t pstride = (size_t)J.kxh * Q;
  load_lines(sm, ldl, np, Q, [&](int l, int p) { return in0[l * pstride + p]; });
  // natural-order input: DIF stages of the inverse leave the rows in DIF
  // order, read back through the position table; DIF-order input: DIT stages
  // leave natural order
  if (J.is_C)
    build_pref_table(tab, J.r + 2 * kPrefWarm + kYChunk, J.box_lo, J.box_len, J.start, Q,
                     J.natural ? J.fy.pos : nullptr, J.periodic != 0);
  __syncthreads();
  if constexpr (FIXP > 0) {
    if (J.natural) fft_smem_plan<kInvDif, FIXP, FixedPlan<FIXP>::L + 1>(sm, np, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
    else fft_smem_plan<kInvDit, FIXP, FixedPlan<FIXP>::L + 1>(sm, np, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
  } else {
    if (J.natural) fft_smem<kInvDif, float2, RSET>(sm, ldl, np, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
    else fft_smem<kInvDit, float2, RSET>(sm, ldl, np, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
  }
  if (!J.is_C) {
    for (int l = 0; l < np; ++l) {
      float2* dst = J.outH + ((size_t)(p0 + l) * J.kxh + kx) * J.ny;
      for (int y = threadIdx.x; y < J.ny; y += blockDim.x)
        dst[y] = sm[l * ldl + (J.natural ? __ldg(J.fy.pos + y) : y)];
    }
    return;
  }
  const int r = J.r;
  if (J.fir) {
    const int nch = (r + kYChunk - 1) / kYChunk;
    for (int i = threadIdx.x; i < np * nch; i += blockDim.x) {
      const int l = i / nch;
      const int k0 = (i - l * nch) * kYChunk;
      const float2* line = sm + l * ldl;
      float2* dst = J.outC + ((size_t)(p0 + l) * J.kxh + kx) * r;
      prefilter_chunk<kYChunk, f2>(
          k0, r, [&](int jj) { return f2(line[tab[jj]]); },
          [&](int k, f2 v) { dst[k] = make_float2(v.x, v.y); });
    }
  } else {
    for (int l = 0; l < np; ++l) {
      float2* dst = J.outC + ((size_t)(p0 + l) * J.kxh + kx) * r;
      for (int k = threadIdx.x; k < r; k += blockDim.x) dst[k] = sm[l * ldl + tab[k + kPrefWarm]];
    }
  }
}

// ------------------------------------------------------------------ direct z sum
// The plane mixing of Sec. III.A for sources of up to kMaxNzDirect layers.
// CTA -> (two kx columns, a chunk of kZMixChunk frequency pairs ky, Qy - ky):
// the input planes of the chunk are staged in shared memory once, both columns
// packed (fft2.cuh), then each warp takes output planes with one frequency pair
// per lane.  A warp takes two coefficient planes, or the three demag planes of
// one layer, at a time: every staged input then serves two or three outputs,
// and the kernel spectra stream through as whole quads (coalesced float4, two
// planes of both columns).
constexpr int kZMixThreads = 128;
constexpr int kZMixChunk = 32;  // frequency pairs per CTA, one per lane

__global__ void __launch_bounds__(kZMixThreads) k_zmix3(const Launch<ZMixJob> Lc) {
  extern __shared__ float4 zs[];  // [2][3 nz][kZMixChunk]: inputs at ky, then at Qy - ky with m_y negated
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const ZMixJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int nch = (J.kyq + kZMixChunk - 1) / kZMixChunk;
  const int kxp = tile / nch;
  const int k0 = (tile - kxp * nch) * kZMixChunk;
  const int nk = min(kZMixChunk, J.kyq - k0);
  const int kxa = 2 * kxp;
  const bool has_b = kxa + 1 < J.kxh;  // an odd last column runs beside itself, stored once
  const int Qy = J.Qy, nz = J.nz, P3 = 3 * nz;
  const size_t pstride = (size_t)J.kxh * Qy;  // one input / output plane
  const int cb = has_b ? Qy : 0;
  const float2* inb = J.in + (size_t)kxa * Qy;
  for (int i = threadIdx.x; i < P3 * kZMixChunk; i += blockDim.x) {
    const int p = i / kZMixChunk, l = i - p * kZMixChunk;
    if (l < nk) {
      const int k = k0 + l;
      const int k1 = k != 0 && 2 * k != Qy ? Qy - k : k;
      const float2* row = inb + (size_t)p * pstride;
      const float2 a = row[k], b = row[k + cb];
      float2 c = row[k1], d = row[k1 + cb];
      if (p >= nz && p < 2 * nz) {  // odd in y: the sums below then need no sign of their own
        c.x = -c.x; c.y = -c.y; d.x = -d.x; d.y = -d.y;
      }
      zs[i] = make_float4(a.x, b.x, a.y, b.y);
      zs[P3 * kZMixChunk + i] = make_float4(c.x, d.x, c.y, d.y);
    }
  }
  __syncthreads();
  const int l = threadIdx.x % kZMixChunk;
  if (l >= nk) return;
  const int k = k0 + l;
  const bool two = k != 0 && 2 * k != Qy;
  const size_t qs = (size_t)((J.kxh + 1) >> 1) * J.kyq;  // quads of two planes
  const size_t koff = (size_t)kxp * J.kyq + k;
  const float4* s0 = zs + l;
  const float4* s1 = zs + P3 * kZMixChunk + l;
  const int kch = (Qy + (int)(kKChunk / 2) - 1) / (int)(kKChunk / 2);
  // value at ky (v0) and at Qy - ky (v1) of plane `o` of an output array
  auto put = [&](float2* out, uint16_t* pk, int o, bool neg1, c2 v0, c2 v1) {
    if (neg1) v1 = c2_scale(p2_dup(-1.f), v1);
    if (pk) {  // reduced precision: straight into the inverse DFT's split operand
      const int prow = o * J.kxh + kxa;
      store_split(pk, kch, prow, k, c2_a(v0));
      if (has_b) store_split(pk, kch, prow + 1, k, c2_b(v0));
      if (two) {
        store_split(pk, kch, prow, Qy - k, c2_a(v1));
        if (has_b) store_split(pk, kch, prow + 1, Qy - k, c2_b(v1));
      }
      return;
    }
    float2* dst = out + (size_t)o * pstride + (size_t)kxa * Qy;
    dst[k] = c2_a(v0);
    if (has_b) dst[k + Qy] = c2_b(v0);
    if (two) {
      dst[Qy - k] = c2_a(v1);
      if (has_b) dst[2 * Qy - k] = c2_b(v1);
    }
  };
  auto in0 = [&](int c, int jz) { return c2_load(s0 + (c * nz + jz) * kZMixChunk); };
  auto in1 = [&](int c, int jz) { return c2_load(s1 + (c * nz + jz) * kZMixChunk); };

  const int npair = (J.n_out + 1) / 2, ndem = J.nH ? nz : 0;
  const int ts2 = t_stride(nz, false) / 2;  // quads per coefficient plane
  for (int task = threadIdx.x / kZMixChunk; task < npair + ndem; task += kZMixThreads / kZMixChunk) {
    if (task < npair) {
      // c(o) = sum_jz sum_c T_c(o, jz) m_c(jz), T_x and T_y imaginary (row z of
      // N too); of the field variant's rows x and y, T_z is the imaginary one
      const int o = 2 * task;
      const bool more = o + 1 < J.n_out;
      const ulonglong2* ta = reinterpret_cast<const ulonglong2*>(J.Tq) + (size_t)o * ts2 * qs + koff;
      const ulonglong2* tb = more ? ta + (size_t)ts2 * qs : ta;
      c2 u[2][2], w[2][2];  // [output][side]: the terms of m_x and m_y, those of m_z
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int s = 0; s < 2; ++s) u[q][s] = w[q][s] = c2_zero();
      auto term = [&](int c, int jz, p2 a, p2 b) {
        const c2 m0 = in0(c, jz), m1 = in1(c, jz);
        c2(*d)[2] = c == 2 ? w : u;
        d[0][0] = c2_axpy(a, m0, d[0][0]);
        d[0][1] = c2_axpy(a, m1, d[0][1]);
        d[1][0] = c2_axpy(b, m0, d[1][0]);
        d[1][1] = c2_axpy(b, m1, d[1][1]);
      };
      int jz = 0;
      for (; jz + 1 < nz; jz += 2) {  // two layers: three quads
        ulonglong2 a[3], b[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          a[q] = __ldg(ta + q * qs);
          b[q] = __ldg(tb + q * qs);
        }
        ta += 3 * qs;
        tb += 3 * qs;
        term(0, jz, a[0].x, b[0].x);
        term(1, jz, a[0].y, b[0].y);
        term(2, jz, a[1].x, b[1].x);
        term(0, jz + 1, a[1].y, b[1].y);
        term(1, jz + 1, a[2].x, b[2].x);
        term(2, jz + 1, a[2].y, b[2].y);
      }
      if (jz < nz) {
        const ulonglong2 a0 = __ldg(ta), a1 = __ldg(ta + qs), b0 = __ldg(tb), b1 = __ldg(tb + qs);
        term(0, jz, a0.x, b0.x);
        term(1, jz, a0.y, b0.y);
        term(2, jz, a1.x, b1.x);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q == 1 && !more) break;
        const int a = J.field_nbox > 0 ? (o + q) / J.field_nbox : 2;
        c2 v[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) v[s] = a == 2 ? c2_add_i<1>(w[q][s], u[q][s]) : c2_add_i<1>(u[q][s], w[q][s]);
        put(J.outC, J.pkC, o + q, a == 1, v[0], v[1]);
      }
    } else {
      // H_a(iz) = sum_jz sum_b Ns_ab(iz - jz) m_b(jz); xz and yz imaginary and odd in dz
      const int iz = task - npair;
      c2 r[3][2], i[3][2];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int s = 0; s < 2; ++s) r[a][s] = i[a][s] = c2_zero();
      for (int jz = 0; jz < nz; ++jz) {
        const int adz = iz >= jz ? iz - jz : jz - iz;
        const ulonglong2* nq = reinterpret_cast<const ulonglong2*>(J.Nq) + (size_t)(3 * adz) * qs + koff;
        const ulonglong2 q0 = __ldg(nq), q1 = __ldg(nq + qs), q2 = __ldg(nq + 2 * qs);
        const p2 sz = p2_dup(iz >= jz ? 1.f : -1.f);
        const p2 xx = q0.x, yy = q0.y, zz = q1.x, xy = q1.y, xz = p2_mul(sz, q2.x), yz = p2_mul(sz, q2.y);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const c2 mx = s ? in1(0, jz) : in0(0, jz), my = s ? in1(1, jz) : in0(1, jz), mz = s ? in1(2, jz) : in0(2, jz);
          r[0][s] = c2_axpy(xy, my, c2_axpy(xx, mx, r[0][s]));
          i[0][s] = c2_axpy(xz, mz, i[0][s]);
          r[1][s] = c2_axpy(yy, my, c2_axpy(xy, mx, r[1][s]));
          i[1][s] = c2_axpy(yz, mz, i[1][s]);
          r[2][s] = c2_axpy(zz, mz, r[2][s]);
          i[2][s] = c2_axpy(yz, my, c2_axpy(xz, mx, i[2][s]));
        }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a)
        put(J.outH, J.pkH, a * nz + iz, a == 1, c2_add_i<1>(r[a][0], i[a][0]), c2_add_i<1>(r[a][1], i[a][1]));
    }
  }
}

// CTAs of a job (the output planes are covered inside each)
int zmix_tiles(int kxh, int kyq) { return (kxh + 1) / 2 * ((kyq + kZMixChunk - 1) / kZMixChunk); }

cudaError_t launch_zmix3(const Launch<ZMixJob>& L, cudaStream_t st) {
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  int nzmax = 1;
  for (int i = 0; i < L.njobs; ++i) nzmax = max(nzmax, L.job[i].nz);
  const size_t smem = sizeof(float4) * 2 * 3 * (size_t)nzmax * kZMixChunk;
  return launch_chained(k_zmix3, grid, kZMixThreads, smem, st, L);
}

// ------------------------------------------------------------------ host side
// about 80 KB of lines per CTA (two CTAs per SM), at least 8 y positions:
// short z grids get many positions, which spreads the per-CTA set-up.  A power
// of two: whole 64-byte runs and no divisions in the output loops.
int zpass_tile(int Qz) {
  const int most = std::max(8, (84 * 1024) / (4 * (Qz + 1) * (int)sizeof(float2)));
  int t = 8;
  while (2 * t <= most) t *= 2;
  return t;
}
int zpass_tiles(int Qy, int ztile) { return (Qy + ztile - 1) / ztile; }

// every job's y plan is 1080 = 12 6 15 (fixed plan 2: the 512 x 512 films)
template <typename JobT> static bool y_fixed_1080(const Launch<JobT>& L) {
  for (int i = 0; i < L.njobs; ++i)
    if (fixed_plan_id(L.job[i].fy.plan) != 2) return false;
  return L.njobs > 0;
}

cudaError_t launch_yfwd3(const Launch<YFwdJob>& L, cudaStream_t st) {
  size_t smem = 0;
  for (int i = 0; i < L.njobs; ++i)
    smem = std::max(smem, sizeof(float2) * (size_t)L.job[i].group * (L.job[i].fy.plan.L + 1));
  unsigned rs = 0;
  for (int i = 0; i < L.njobs; ++i) rs |= plan_radix_set(L.job[i].fy.plan);
  auto k = y_fixed_1080(L) ? k_yfwd3<kAllRadices, 2>
           : (rs & ~kRadixSetA) == 0u ? k_yfwd3<kRadixSetA, 0> : k_yfwd3<kAllRadices, 0>;
  cudaError_t e = allow_smem((const void*)k, 227 * 1024);
  if (e != cudaSuccess) return e;
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  return launch_chained(k, grid, 256, smem, st, L);
}

cudaError_t launch_zpass3(const Launch<ZJob>& L, cudaStream_t st) {
  size_t smem = 0;
  for (int i = 0; i < L.njobs; ++i) {
    const ZJob& J = L.job[i];
    const size_t lines = sizeof(float2) * 4 * J.ztile * (size_t)(J.fz.plan.L + 1);
    const size_t tab = sizeof(int) * (size_t)(J.do_C ? J.r + 2 * kPrefWarm + kZChunk : 0);
    smem = std::max(smem, lines + tab);
  }
  unsigned rs = 0;
  for (int i = 0; i < L.njobs; ++i) rs |= plan_radix_set(L.job[i].fz.plan);
  auto k = (rs & ~kRadixSetA) == 0u ? k_zpass3<kRadixSetA> : k_zpass3<kAllRadices>;
  cudaError_t e = allow_smem((const void*)k, 227 * 1024);
  if (e != cudaSuccess) return e;
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  return launch_chained(k, grid, 256, smem, st, L);
}

cudaError_t launch_yinv3(const Launch<YInvJob>& L, cudaStream_t st) {
  size_t smem = 0;
  for (int i = 0; i < L.njobs; ++i) {
    const YInvJob& J = L.job[i];
    const size_t lines = sizeof(float2) * (size_t)J.group * (J.fy.plan.L + 1);
    const size_t tab = sizeof(int) * (size_t)(J.is_C ? J.r + 2 * kPrefWarm + kYChunk : 0);
    smem = std::max(smem, lines + tab);
  }
  unsigned rs = 0;
  for (int i = 0; i < L.njobs; ++i) rs |= plan_radix_set(L.job[i].fy.plan);
  auto k = y_fixed_1080(L) ? k_yinv3<kAllRadices, 2>
           : (rs & ~kRadixSetA) == 0u ? k_yinv3<kRadixSetA, 0> : k_yinv3<kAllRadices, 0>;
  cudaError_t e = allow_smem((const void*)k, 227 * 1024);
  if (e != cudaSuccess) return e;
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  return launch_chained(k, grid, 256, smem, st, L);
}

}  // namespace mm
