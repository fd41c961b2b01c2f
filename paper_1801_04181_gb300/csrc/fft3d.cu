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
// Two neighbouring y positions are a pair of lines per component (fft2.cuh).
constexpr int kZThreads = 384;  // two CTAs per SM
template <typename Fft>
__global__ void __launch_bounds__(kZThreads, 2) k_zpass3(const Launch<ZJob> Lc) {
  extern __shared__ float4 sm4[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const ZJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int Qy = J.fy.plan.L, Qz = Fft::kL ? Fft::kL : J.fz.plan.L;
  const int zt = J.ztile;
  const int zl = 31 - __clz(zt);  // zt is a power of two
  const int npt = (Qy + zt - 1) >> zl;
  const int kx = tile / npt;
  const int y0 = (tile - kx * npt) << zl;
  const int nt = min(zt, Qy - y0);  // even, as Qy is
  const int np = nt >> 1;           // pairs of positions
  const int nz = J.nz, P3 = 3 * nz;
  const int ldz = Qz + 1;
  // lines: pair * 3 + c (input, then H in place), then the phi line of each pair
  const int nin = 3 * np;
  float4* phi = sm4 + nin * ldz;
  float4* tws = sm4 + 2 * zt * ldz;
  int* tab = reinterpret_cast<int*>(tws + J.fz.ntw2);

  // the 3 nz values of a y position are one run in memory, nz of each
  // component; layers [nz, Qz) are zero padding
  const float2* src = J.in + ((size_t)kx * Qy + y0) * P3;
  Fft::in(
      sm4, ldz, nin, J.fz, tws,
      [&](int l, int z0, int M, auto& v) {
        const int tp = l / 3, c = l - 3 * tp;
        const float2* a = src + (size_t)(2 * tp) * P3 + c * nz + z0;
#pragma unroll
        for (int k = 0; k < (int)(sizeof(v) / sizeof(v[0])); ++k)
          v[k] = z0 + k * M < nz ? c2_make(__ldg(a + k * M), __ldg(a + k * M + P3)) : c2_zero();
      },
      [&]() {
        for (int i = threadIdx.x; i < J.fz.ntw2; i += blockDim.x) tws[i] = __ldg(J.fz.tw2 + i);
        if (J.do_C)
          build_pref_table(tab, J.r + 2 * kPrefWarm + kZChunk, J.box_lo, J.box_len, J.start, Qz, nullptr);
      });

  // spectral products at the pair (kz, Qz - kz): lanes along kz, warps along
  // the position pairs
  const int half = Qz >> 1;
  const size_t kstride = (size_t)J.kxh * J.kyq * J.kzq;
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int runs = (half + 32) >> 5;
  for (int task = threadIdx.x >> 5; task < np * runs; task += warps) {
    const int tp = task / runs, kz = ((task - tp * runs) << 5) + lane;
    if (kz > half) continue;
    const int kya = __ldg(J.fy.freq + y0 + 2 * tp), kyb = __ldg(J.fy.freq + y0 + 2 * tp + 1);
    const bool ma = 2 * kya > Qy, mb = 2 * kyb > Qy;
    const p2 sy = p2_pack(ma ? -1.f : 1.f, mb ? -1.f : 1.f), minus = p2_dup(-1.f);
    const size_t oa = ((size_t)kx * J.kyq + (ma ? Qy - kya : kya)) * J.kzq + kz;
    const size_t ob = ((size_t)kx * J.kyq + (mb ? Qy - kyb : kyb)) * J.kzq + kz;
    p2 nv[6], sv[3];
#pragma unroll
    for (int c = 0; c < 6; ++c)
      nv[c] = J.do_H ? p2_pack(__ldg(J.N3 + c * kstride + oa), __ldg(J.N3 + c * kstride + ob)) : 0ull;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      sv[c] = J.do_C ? p2_pack(__ldg(J.S3 + c * kstride + oa), __ldg(J.S3 + c * kstride + ob)) : 0ull;
    // odd in y: S_y, N_xy, N_yz; odd in z (negated at Qz - kz): S_z, N_xz, N_yz
    sv[1] = p2_mul(sy, sv[1]);
    nv[3] = p2_mul(sy, nv[3]);
    nv[5] = p2_mul(sy, nv[5]);
    const bool two = kz != 0 && 2 * kz != Qz;
    float4* line = sm4 + 3 * tp * ldz;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (side == 1) {
        if (!two) break;
        sv[2] = p2_mul(minus, sv[2]);
        nv[4] = p2_mul(minus, nv[4]);
        nv[5] = p2_mul(minus, nv[5]);
      }
      const int q = __ldg(J.fz.pos + (side ? Qz - kz : kz));
      const c2 mx = c2_load(line + q), my = c2_load(line + ldz + q), mz = c2_load(line + 2 * ldz + q);
      if (J.do_C) {  // phi = i (Sx mx + Sy my + Sz mz)
        const c2 s = c2_axpy(sv[0], mx, c2_axpy(sv[1], my, c2_scale(sv[2], mz)));
        c2_store(phi + tp * ldz + q, c2_rot4<1>(s));
      }
      if (J.do_H) {  // N real
        c2_store(line + q, c2_axpy(nv[0], mx, c2_axpy(nv[3], my, c2_scale(nv[4], mz))));
        c2_store(line + ldz + q, c2_axpy(nv[3], mx, c2_axpy(nv[1], my, c2_scale(nv[5], mz))));
        c2_store(line + 2 * ldz + q, c2_axpy(nv[4], mx, c2_axpy(nv[5], my, c2_scale(nv[2], mz))));
      }
    }
  }
  __syncthreads();
  {
    float4* first = J.do_H ? sm4 : phi;
    Fft::out(first, ldz, (J.do_H ? nin : 0) + (J.do_C ? np : 0), J.fz, tws, [&](int l, int z0, int M, auto& v) {
      float4* p = first + (l * ldz + z0);
#pragma unroll
      for (int k = 0; k < (int)(sizeof(v) / sizeof(v[0])); ++k) c2_store(p + k * M, v[k]);
    });
  }

  // outputs with the y position fastest: runs of the tile's positions
  const int pl = zl - 1;  // log2 of the pairs of a whole tile
  if (J.do_H) {
    for (int c = 0; c < 3; ++c) {
      float2* out = J.outH + ((size_t)c * nz * J.kxh + kx) * Qy + y0;
      for (int i = threadIdx.x; i < nz << pl; i += blockDim.x) {
        const int z = i >> pl, tp = i & ((1 << pl) - 1);
        if (tp >= np) continue;
        const float4 v = sm4[(tp * 3 + c) * ldz + z];
        *reinterpret_cast<float4*>(out + (size_t)z * J.kxh * Qy + 2 * tp) = make_float4(v.x, v.z, v.y, v.w);
      }
    }
  }
  if (J.do_C) {
    const int r = J.r;
    float2* out = J.outC + (size_t)kx * Qy + y0;
    const size_t ostride = (size_t)J.kxh * Qy;
    if (J.fir) {
      // one thread per chunk and per real or imaginary part (of both
      // positions); the two parts swap halves to store whole values
      const int nch = (r + kZChunk - 1) / kZChunk;
      const int items = nch << zl;
      for (int base = threadIdx.x & ~31; base < items; base += blockDim.x) {
        const int idx = min(base + lane, items - 1);  // whole warps swap (items is even)
        const int part = idx & 1, tp = (idx >> 1) & ((1 << pl) - 1);
        const int k0 = (idx >> zl) * kZChunk;
        const bool store = base + lane < items && tp < np;
        const p2* line = reinterpret_cast<const p2*>(phi + min(tp, np - 1) * ldz) + part;
        float2* dst = out + 2 * tp + part;
        prefilter_chunk2<kZChunk>(
            k0, [&](int jj) { return line[2 * tab[jj]]; },
            [&](int k, p2 v) {
              const float2 f = p2_unpack(v);  // (position a, position b) of this part
              const float other = __shfl_xor_sync(0xffffffffu, part ? f.x : f.y, 1);
              if (store && k < r) dst[k * ostride] = part ? make_float2(other, f.y) : make_float2(f.x, other);
            });
      }
    } else {
      for (int i = threadIdx.x; i < r << pl; i += blockDim.x) {
        const int k = i >> pl, tp = i & ((1 << pl) - 1);
        if (tp >= np) continue;
        const float4 v = phi[tp * ldz + tab[k + kPrefWarm]];
        *reinterpret_cast<float4*>(out + k * ostride + 2 * tp) = make_float4(v.x, v.z, v.y, v.w);
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
// of two: whole 64-byte runs and no divisions in the output loops.  Four where
// the longest lines leave no room for the twiddles (at most 2 Qz) and the
// prefilter table (at most Qz + 37).
int zpass_tile(int Qz) {
  const int most = std::max(8, (84 * 1024) / (4 * (Qz + 1) * (int)sizeof(float2)));
  int t = 8;
  while (2 * t <= most) t *= 2;
  const size_t tables = 2 * sizeof(float4) * (size_t)Qz + sizeof(int) * (size_t)(Qz + 2 * kPrefWarm + kZChunk);
  if (2 * sizeof(float4) * (size_t)t * (Qz + 1) + tables > 227 * 1024) t = 4;
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

// the lengths of 64 and 128 layers, their plans as constants: 64 x 64 x 64 228 -> 209
// us, 64 x 64 x 128 427 -> 391 us a launch
using ZPairPlans = PairPlans<CtPair<4, 8, 5, 1, 1>, CtPair<4, 8, 9, 1, 1>>;
struct ZPass3 {
  static constexpr bool takes(int) { return true; }
  template <typename Fft> static auto build() { return &k_zpass3<Fft>; }
};

cudaError_t launch_zpass3(const Launch<ZJob>& L, cudaStream_t st) {
  size_t smem = 0;
  for (int i = 0; i < L.njobs; ++i) {
    const ZJob& J = L.job[i];
    const FftPlanDev& P = J.fz.plan;
    const size_t lines = sizeof(float4) * (2 * J.ztile * (size_t)(P.L + 1) + J.fz.ntw2);
    const size_t tab = sizeof(int) * (size_t)(J.do_C ? J.r + 2 * kPrefWarm + kZChunk : 0);
    smem = std::max(smem, lines + tab);
  }
  auto k = ZPairPlans::kernel<ZPass3>(L, &ZJob::fz);
  cudaError_t e = allow_smem((const void*)k, 227 * 1024);
  if (e != cudaSuccess) return e;
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  return launch_chained(k, grid, kZThreads, smem, st, L);
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
