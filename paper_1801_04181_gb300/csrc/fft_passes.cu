// FFT passes of the potential / self-demag convolution (Sec. III.A).
//
// Per source magnet s the circular convolution over a Qx x Qy grid runs as
//   x pass (R2C, two real rows per complex line)  -> X1[plane][kx][y]
//   y pass: forward y FFT, z plane mixing with the kernel spectra, inverse y
//           FFT, y prefilter of the coefficient planes    -> Y[plane][kx][row]
//   x pass (C2R, two rows per line), x prefilter          -> real rows
// Spectra are stored kx-major with y fastest, so every pass reads and writes
// whole contiguous rows or columns of HBM.  Thin films (nz <= 4) take z by a
// direct sum over planes inside the y pass, which saves a third FFT pass.
//
// Kernel spectra are real quarter planes (kx <= Qx/2, ky <= Qy/2): every
// component of S and N is even or odd in x and y, so its spectrum is purely
// real or purely imaginary and even or odd in ky.  Signs and the factor i are
// restored here; one thread handles the pair (ky, Qy - ky), which shares the
// stored values, and walks ky in natural order so those loads coalesce.
// Thicker magnets (nz > 4) take z by an FFT pass of its own (fft3d.cu).
#include "fft.cuh"
#include "fft2.cuh"
#include "mm_internal.h"
#include "prefilter.cuh"
#include "umma.cuh"

namespace mm {

constexpr int kLines = kRowsPerCta / 2;  // complex lines per CTA in the x passes
// threads per CTA of the x passes (multiples of kLines)
constexpr int kXFwdThreads = 256;
constexpr int kXInvThreads = 256;
constexpr int kLinePad = 4;              // float2 between lines of an x-pass CTA

cudaError_t init_fft_constants_passes() { return upload_roots(); }

// ------------------------------------------------------------------ x forward
// FIXP > 0: every job's x plan is fixed plan FIXP, run with its lengths as constants.
template <unsigned RSET, int FIXP>
__global__ void __launch_bounds__(kXFwdThreads, 3) k_xfwd(const Launch<XFwdJob> Lc) {
  extern __shared__ float2 sm[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const XFwdJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int Q = FIXP ? FixedPlan<FIXP ? FIXP : 1>::L : J.fx.plan.L;
  const int ldl = Q + kLinePad;  // padded line stride: the lines start in different banks
  const int rows = 3 * J.nz * J.ny;
  const int r0 = tile * kRowsPerCta;
  const int nrows = min(kRowsPerCta, rows - r0);
  const int nlines = (nrows + 1) >> 1;
  const int nx = J.nx;
  const float* row0 = J.m + (size_t)r0 * nx;

  if ((nx & 3) == 0) {
    // all rows of the CTA per thread and step: 2 kLines float4 loads in flight
    const int n4 = nx >> 2;
    for (int x4 = threadIdx.x; x4 < n4; x4 += blockDim.x) {
      float4 v[kRowsPerCta];
#pragma unroll
      for (int r = 0; r < kRowsPerCta; ++r)
        v[r] = r < nrows ? __ldg(reinterpret_cast<const float4*>(row0 + r * nx) + x4)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int l = 0; l < kLines; ++l) {
        if (l < nlines) {
          float2* d = sm + l * ldl + 4 * x4;
          const float4 a = v[2 * l], b = v[2 * l + 1];
          d[0] = make_float2(a.x, b.x);
          d[1] = make_float2(a.y, b.y);
          d[2] = make_float2(a.z, b.z);
          d[3] = make_float2(a.w, b.w);
        }
      }
    }
  } else {
    for (int x = threadIdx.x; x < nx; x += blockDim.x) {
      float v[kRowsPerCta];
#pragma unroll
      for (int r = 0; r < kRowsPerCta; ++r) v[r] = r < nrows ? __ldg(row0 + r * nx + x) : 0.f;
#pragma unroll
      for (int l = 0; l < kLines; ++l)
        if (l < nlines) sm[l * ldl + x] = make_float2(v[2 * l], v[2 * l + 1]);
    }
  }
  // entries [nx, Q) are zero padding: the first stage takes them as zero unread
  // DIF positions of k and Q - k for every kx <= Q/2
  ushort2* ptab = reinterpret_cast<ushort2*>(sm + kLines * ldl);  // Q < 65536
  for (int kx = threadIdx.x; kx < J.kxh; kx += blockDim.x)
    ptab[kx] = make_ushort2((unsigned short)__ldg(J.fx.pos + kx),
                            (unsigned short)__ldg(J.fx.pos + (kx == 0 ? 0 : Q - kx)));
  __syncthreads();
  if constexpr (FIXP > 0)
    fft_smem_plan<kFwdDif, FIXP, FixedPlan<FIXP>::L + kLinePad>(sm, nlines, J.fx.plan, J.fx.tw_f, 0, blockDim.x, nx);
  else
    fft_smem<kFwdDif, float2, RSET>(sm, ldl, nlines, J.fx.plan, J.fx.tw_f, 0, blockDim.x, nx);

  // Z = A + iB:  A_k = (Z_k + conj Z_{Q-k}) / 2,  B_k = (Z_k - conj Z_{Q-k}) / (2i)
  // thread -> (kx, line) with the line fastest: a warp writes 8 runs of 64 bytes
  const int ny = J.ny;
  const int pa0 = r0 / ny;
  const bool pairs = (ny & 1) == 0 && (nrows & 1) == 0;  // both rows of a line in one plane, 16-B aligned
  if (pairs && nlines == kLines) {
    // full tile: blockDim is a multiple of kLines, so every thread keeps one
    // line and its output row pair for all its kx
    const int l = threadIdx.x % kLines;
    int pa = pa0, ya = r0 + 2 * l - pa0 * ny;
    while (ya >= ny) { ++pa; ya -= ny; }
    float2* dst0 = J.out + (size_t)pa * J.kxh * ny + ya;
    const float2* line = sm + l * ldl;
    const int kch = (ny + (int)(kKChunk / 2) - 1) / (int)(kKChunk / 2);
    for (int kx = threadIdx.x / kLines; kx < J.kxh; kx += blockDim.x / kLines) {
      const ushort2 pp = ptab[kx];
      const float2 Zk = line[pp.x];
      const float2 Zm = line[pp.y];
      if (J.pk) {  // reduced precision: straight into the forward DFT's split operand
        store_split(J.pk, kch, pa * J.kxh + kx, ya, make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y - Zm.y)));
        store_split(J.pk, kch, pa * J.kxh + kx, ya + 1, make_float2(0.5f * (Zk.y + Zm.y), -0.5f * (Zk.x - Zm.x)));
      } else {
        *reinterpret_cast<float4*>(dst0 + (size_t)kx * ny) =
            make_float4(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y - Zm.y), 0.5f * (Zk.y + Zm.y), -0.5f * (Zk.x - Zm.x));
      }
    }
    return;
  }
  const int n = J.kxh * nlines;
  for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
    const int kx = nlines == kLines ? idx / kLines : idx / nlines;
    const int l = idx - kx * nlines;
    const ushort2 pp = ptab[kx];
    const float2 Zk = sm[l * ldl + pp.x];
    const float2 Zm = sm[l * ldl + pp.y];
    const float2 A = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y - Zm.y));
    const float2 B = make_float2(0.5f * (Zk.y + Zm.y), -0.5f * (Zk.x - Zm.x));
    int pa = pa0, ya = r0 + 2 * l - pa0 * ny;
    while (ya >= ny) { ++pa; ya -= ny; }
    if (J.pk) {
      const int kch = (ny + (int)(kKChunk / 2) - 1) / (int)(kKChunk / 2);
      store_split(J.pk, kch, pa * J.kxh + kx, ya, A);
      if (2 * l + 1 < nrows) {
        int pb = pa, yb = ya + 1;
        if (yb >= ny) { ++pb; yb -= ny; }
        store_split(J.pk, kch, pb * J.kxh + kx, yb, B);
      }
      continue;
    }
    float2* dst = J.out + ((size_t)pa * J.kxh + kx) * ny + ya;
    if (pairs) {
      *reinterpret_cast<float4*>(dst) = make_float4(A.x, A.y, B.x, B.y);
    } else {
      *dst = A;
      if (2 * l + 1 < nrows) {
        int pb = pa, yb = ya + 1;
        if (yb >= ny) { ++pb; yb -= ny; }
        J.out[((size_t)pb * J.kxh + kx) * ny + yb] = B;
      }
    }
  }
}

// ------------------------------------------------------------------ y pass
__device__ __forceinline__ float2 kmul(float v, bool imag, float2 m) {
  return imag ? make_float2(-v * m.y, v * m.x) : make_float2(v * m.x, v * m.y);
}
__device__ __forceinline__ void cacc(float2& a, float2 b) { a.x += b.x; a.y += b.y; }

template <int NZ>
__device__ __forceinline__ void load_pair(const float2* sm, int Q, int p0, int p1, float2 (*mh)[3][NZ]) {
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
      mh[0][c][z] = sm[(c * NZ + z) * Q + p0];
      mh[1][c][z] = sm[(c * NZ + z) * Q + p1];
    }
}

// Spectral products at every (ky, Qy - ky) pair of one kx column.  The
// potential planes land beyond the input planes whenever the demag planes are
// produced too; those overwrite the inputs in place.  A thread owns the two
// positions of its pair in every plane, so it reads the inputs once and writes
// both products without any barrier.  Kernel-spectrum loads are issued in
// batches before the arithmetic that uses them.
template <int NZ>
__device__ __forceinline__ void ypass_mix(const YJob& J, float2* sm, int kx, int Q, int nH) {
  // output planes per batch of kernel loads (about 30 values in flight)
  constexpr int OB = 30 / (3 * NZ) > 0 ? 30 / (3 * NZ) : 1;
  const int kstride = J.kxh * J.kyq;  // one stored kernel plane (< 2^31 values in all)
  const int half = Q >> 1;
  for (int kyq = threadIdx.x; kyq <= half; kyq += blockDim.x) {
    // the two frequencies ky = kyq and Qy - kyq share every stored kernel value;
    // the second has the odd-in-y components negated
    const bool two = kyq != 0 && 2 * kyq != Q;
    const int koff = kx * J.kyq + kyq;
    const int p0 = fft_pos(kyq, J.fy.plan);
    const int p1 = two ? fft_pos(Q - kyq, J.fy.plan) : p0;
    float2 mh[2][3][NZ];
    load_pair<NZ>(sm, Q, p0, p1, mh);
    if (J.do_C) {
      const float* Tk = J.Tq + koff;
      for (int ob = 0; ob < J.n_out; ob += OB) {
        float tv[OB][NZ][3];
#pragma unroll
        for (int o = 0; o < OB; ++o)
#pragma unroll
          for (int jz = 0; jz < NZ; ++jz)
#pragma unroll
            for (int c = 0; c < 3; ++c)
              tv[o][jz][c] = ob + o < J.n_out ? __ldg(Tk + (((ob + o) * NZ + jz) * 3 + c) * kstride) : 0.f;
        // c(o) = sum_jz sum_c T_c(o, jz) m_c(jz); T = Ms W (S spectra) / (Qx Qy)
#pragma unroll
        for (int o = 0; o < OB; ++o) {
          if (ob + o >= J.n_out) break;
          float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
#pragma unroll
          for (int jz = 0; jz < NZ; ++jz) {
            const float tx = tv[o][jz][0], ty = tv[o][jz][1], tz = tv[o][jz][2];
            cacc(acc0, kmul(tx, true, mh[0][0][jz]));
            cacc(acc0, kmul(ty, true, mh[0][1][jz]));
            cacc(acc0, kmul(tz, false, mh[0][2][jz]));
            cacc(acc1, kmul(tx, true, mh[1][0][jz]));
            cacc(acc1, kmul(-ty, true, mh[1][1][jz]));
            cacc(acc1, kmul(tz, false, mh[1][2][jz]));
          }
          sm[(nH + ob + o) * Q + p0] = acc0;
          if (two) sm[(nH + ob + o) * Q + p1] = acc1;
        }
      }
    }
    if (J.do_H) {
      // H_a(iz) = sum_jz sum_b Ns_ab(iz - jz) m_b(jz); Ns = -Ms N / (Qx Qy)
      const float* Nk = J.Nq + koff;
      float nv[6][NZ];
#pragma unroll
      for (int comp = 0; comp < 6; ++comp)
#pragma unroll
        for (int dz = 0; dz < NZ; ++dz) nv[comp][dz] = __ldg(Nk + (dz * 6 + comp) * kstride);
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const float fy = side ? -1.f : 1.f;
        const int p = side ? p1 : p0;
        if (side == 1 && !two) break;
#pragma unroll
        for (int iz = 0; iz < NZ; ++iz) {
          float2 a0 = make_float2(0.f, 0.f), a1 = a0, a2 = a0;
#pragma unroll
          for (int jz = 0; jz < NZ; ++jz) {
            const int adz = iz >= jz ? iz - jz : jz - iz;
            const float sz = iz >= jz ? 1.f : -1.f;
            const float nxx = nv[0][adz], nyy = nv[1][adz], nzz = nv[2][adz];
            const float nxy = nv[3][adz] * fy, nxz = nv[4][adz] * sz, nyz = nv[5][adz] * sz * fy;
            const float2 mx = mh[side][0][jz], my = mh[side][1][jz], mz = mh[side][2][jz];
            cacc(a0, kmul(nxx, false, mx)); cacc(a0, kmul(nxy, false, my)); cacc(a0, kmul(nxz, true, mz));
            cacc(a1, kmul(nxy, false, mx)); cacc(a1, kmul(nyy, false, my)); cacc(a1, kmul(nyz, true, mz));
            cacc(a2, kmul(nxz, true, mx));  cacc(a2, kmul(nyz, true, my));  cacc(a2, kmul(nzz, false, mz));
          }
          sm[(0 * NZ + iz) * Q + p] = a0;
          sm[(1 * NZ + iz) * Q + p] = a1;
          sm[(2 * NZ + iz) * Q + p] = a2;
        }
      }
    }
  }
}

// One column per CTA (ypass_pairs: where two do not pay); kernel spectra by planes.  Every job of a launch has NZ layers.  kYThreads = 288 (nine
// warps) covers the 271 frequency pairs of a 540-point line in one round of
// the spectral products.
constexpr int kYThreads = 288;
// FIX540: every job's y plan is 540 = 4 9 15, run with its lengths as constants.
template <int NZ, unsigned RSET, bool FIX540>
__global__ void __launch_bounds__(kYThreads, NZ <= 2 ? 3 : 2) k_ypass(const Launch<YJob> Lc) {
  constexpr int Pin = 3 * NZ;
  extern __shared__ float2 sm[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const YJob& J = Lc.job[j];
  const int kx = blockIdx.x - Lc.tile_start[j];
  const int Q = J.fy.plan.L;
  const int nH = J.do_H ? Pin : 0;
  const int Pout = nH + (J.do_C ? J.n_out : 0);
  int* tab = reinterpret_cast<int*>(sm + max(Pin, Pout) * Q);
  const int ny = J.ny;
  const float2* col0 = J.in + (size_t)kx * ny;
  const size_t pstride = (size_t)J.kxh * ny;  // one input plane

  // The kernel spectra of this kx column are read only after the forward FFT:
  // start moving their lines into L2 now (one prefetch per 128-byte line).
  {
    const size_t kstride = (size_t)J.kxh * J.kyq;
    const int lines = (J.kyq + 31) / 32;
    const int nN = J.do_H ? 6 * NZ : 0;
    const int nT = J.do_C ? 3 * NZ * J.n_out : 0;
    for (int i = threadIdx.x; i < (nN + nT) * lines; i += blockDim.x) {
      const int row = i / lines, ln = i - row * lines;
      const float* p = row < nN ? J.Nq + (size_t)row * kstride : J.Tq + (size_t)(row - nN) * kstride;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(p + (size_t)kx * J.kyq + 32 * ln));
    }
  }

  if ((ny & 1) == 0) {
    // one float4 (two complex rows) of every plane per thread and step
    const int n2 = ny >> 1;
    for (int y2 = threadIdx.x; y2 < n2; y2 += blockDim.x) {
      float4 v[Pin];
#pragma unroll
      for (int p = 0; p < Pin; ++p) v[p] = *(reinterpret_cast<const float4*>(col0 + p * pstride) + y2);
#pragma unroll
      for (int p = 0; p < Pin; ++p) {
        sm[p * Q + 2 * y2] = make_float2(v[p].x, v[p].y);
        sm[p * Q + 2 * y2 + 1] = make_float2(v[p].z, v[p].w);
      }
    }
  } else {
    for (int y = threadIdx.x; y < ny; y += blockDim.x) {
      float2 v[Pin];
#pragma unroll
      for (int p = 0; p < Pin; ++p) v[p] = col0[p * pstride + y];
#pragma unroll
      for (int p = 0; p < Pin; ++p) sm[p * Q + y] = v[p];
    }
  }
  // (taking the zero rows as zero unread in the first stage measured slower here)
  for (int y = ny + threadIdx.x; y < Q; y += blockDim.x)
#pragma unroll
    for (int p = 0; p < Pin; ++p) sm[p * Q + y] = make_float2(0.f, 0.f);
  if (J.do_C)
    build_pref_table(tab, J.r + 2 * kPrefWarm + kYChunk, J.box_lo, J.box_len, J.start, Q, nullptr, J.periodic != 0);
  __syncthreads();
  if constexpr (FIX540) fft_smem_fixed<kFwdDif, float2, 4, 9, 15>(sm, Pin, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
  else fft_smem<kFwdDif, float2, RSET>(sm, Q, Pin, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
  ypass_mix<NZ>(J, sm, kx, Q, nH);
  __syncthreads();
  if constexpr (FIX540) fft_smem_fixed<kInvDit, float2, 4, 9, 15>(sm, Pout, J.fy.plan, J.fy.tw_f, 0, blockDim.x);
  else fft_smem<kInvDit, float2, RSET>(sm, Q, Pout, J.fy.plan, J.fy.tw_f, 0, blockDim.x);

  if (J.do_H) {
    float2* out0 = J.outH + (size_t)kx * ny;
    for (int y = threadIdx.x; y < ny; y += blockDim.x)
#pragma unroll
      for (int p = 0; p < Pin; ++p) out0[p * pstride + y] = sm[p * Q + y];
  }
  if (J.do_C) {
    const int r = J.r;
    float2* out0 = J.outC + (size_t)kx * r;
    const size_t ostride = (size_t)J.kxh * r;
    if (J.fir) {
      const int nch = (r + kYChunk - 1) / kYChunk;
      for (int idx = threadIdx.x; idx < J.n_out * nch; idx += blockDim.x) {
        const int o = idx / nch;
        const int k0 = (idx - o * nch) * kYChunk;
        const float2* col = sm + (nH + o) * Q;
        float2* dst = out0 + o * ostride;
        prefilter_chunk<kYChunk, f2>(
            k0, r, [&](int jj) { return f2(col[tab[jj]]); },
            [&](int k, f2 v) { dst[k] = make_float2(v.x, v.y); });
      }
    } else {
      for (int k = threadIdx.x; k < r; k += blockDim.x) {
        const int t = tab[k + kPrefWarm];
        for (int o = 0; o < J.n_out; ++o) out0[o * ostride + k] = sm[(nH + o) * Q + t];
      }
    }
  }
}

// ------------------------------------------------------------------ y pass, two columns per CTA
// The same pass on the columns kx and kx + 1 as one pair of lines per plane
// (fft2.cuh): transforms, spectral products and the prefilter run both columns
// in packed arithmetic.

// Spectral products of the coefficient planes [c0, c1) (placed from plane cb
// on) and, last, of the demag planes, at every (ky, Qy - ky) pair.  Terms whose
// kernel spectrum is real and those whose spectrum is imaginary are summed
// apart and the factor i is applied once; at Qy - ky the components odd in y
// change sign, which is the same as negating m_y there and H_y in the result.
// One thread per frequency of a pair (neighbouring lanes: their loads
// coincide); the kernel values come as quads, both columns packed.
template <int NZ>
__device__ __forceinline__ void ypass2_mix(const YJob& J, float4* sm, int kxp, int Q, int cb, int c0, int c1,
                                           bool do_H) {
  constexpr int TS = t_stride(NZ, true);
  static_assert(NZ <= 3, "four layers run one column per CTA");
  constexpr int OB = NZ == 1 ? 4 : NZ == 2 ? 3 : 1;  // outputs per batch of loads: whole quads
  constexpr int TQ = (OB * TS + 1) / 2;    // their quads
  const unsigned qs = (unsigned)((J.kxh + 1) >> 1) * J.kyq;  // quads of two planes
  const p2 minus = p2_dup(-1.f);
  for (int item = threadIdx.x; item < 2 * J.kyq; item += blockDim.x) {
    const int kyq = item >> 1;
    const bool mirror = (item & 1) != 0;  // this thread's frequency is Qy - kyq
    if (mirror && (kyq == 0 || 2 * kyq == Q)) continue;
    float4* at = sm + __ldg(J.fy.pos + (mirror ? Q - kyq : kyq));
    c2 mh[3][NZ];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int z = 0; z < NZ; ++z) mh[c][z] = c2_load(at + (c * NZ + z) * Q);
    if (mirror)
#pragma unroll
      for (int z = 0; z < NZ; ++z) mh[1][z] = c2_scale(minus, mh[1][z]);
    const unsigned koff = (unsigned)kxp * J.kyq + kyq;
    const ulonglong2* Tk = reinterpret_cast<const ulonglong2*>(J.Tq) + koff;
    for (int ob = c0; ob < c1; ob += OB) {
      p2 tv[2 * TQ];
#pragma unroll
      for (int q = 0; q < TQ; ++q) {
        // quads of outputs past the last are not read (a batch starts on a whole quad)
        if (ob + (2 * q) / TS < c1) {
          const ulonglong2 v = __ldg(Tk + (size_t)(ob * TS / 2 + q) * qs);
          tv[2 * q] = v.x; tv[2 * q + 1] = v.y;
        } else {
          tv[2 * q] = tv[2 * q + 1] = 0ull;
        }
      }
      // c(o) = sum_jz sum_c T_c(o, jz) m_c(jz); T_x, T_y imaginary, T_z real
#pragma unroll
      for (int o = 0; o < OB; ++o) {
        if (ob + o >= c1) break;
        const p2* t = tv + o * TS;
        c2 r = c2_scale(t[2], mh[2][0]), i = c2_scale(t[0], mh[0][0]);
        i = c2_axpy(t[1], mh[1][0], i);
#pragma unroll
        for (int jz = 1; jz < NZ; ++jz) {
          r = c2_axpy(t[3 * jz + 2], mh[2][jz], r);
          i = c2_axpy(t[3 * jz], mh[0][jz], i);
          i = c2_axpy(t[3 * jz + 1], mh[1][jz], i);
        }
        c2_store(at + (cb + ob + o - c0) * Q, c2_add_i<1>(r, i));
      }
    }
    if (!do_H) continue;
    // H_a(iz) = sum_jz sum_b Ns_ab(iz - jz) m_b(jz), the planes dz * 6 + (xx yy
    // zz xy xz yz); xz and yz imaginary and odd in dz
    const ulonglong2* Nk = reinterpret_cast<const ulonglong2*>(J.Nq) + koff;
    p2 nv[6 * NZ];
#pragma unroll
    for (int q = 0; q < 3 * NZ; ++q) {
      const ulonglong2 v = __ldg(Nk + (size_t)q * qs);
      nv[2 * q] = v.x; nv[2 * q + 1] = v.y;
    }
#pragma unroll
    for (int iz = 0; iz < NZ; ++iz) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        c2 r = c2_zero(), ip = r, im = r;  // real terms; imaginary ones with dz >= 0 and dz < 0
#pragma unroll
        for (int jz = 0; jz < NZ; ++jz) {
          const int adz = iz >= jz ? iz - jz : jz - iz;
#pragma unroll
          for (int b = 0; b < 3; ++b) {
            const int comp = a == b ? a : a + b + 2;
            const bool imag = (a == 2) != (b == 2);
            if (!imag) r = c2_axpy(nv[adz * 6 + comp], mh[b][jz], r);
            else if (iz >= jz) ip = c2_axpy(nv[adz * 6 + comp], mh[b][jz], ip);
            else im = c2_axpy(nv[adz * 6 + comp], mh[b][jz], im);
          }
        }
        c2 h = c2_add_i<1>(r, iz + 1 < NZ ? ip - im : ip);  // no dz < 0 term in the last layer
        if (a == 1 && mirror) h = c2_scale(minus, h);
        c2_store(at + (a * NZ + iz) * Q, h);
      }
    }
  }
}

// Planes of a CTA in shared memory: the 3 NZ input planes (then the demag
// planes, in place) and `ch` coefficient planes at a time.
//
// What bounds it: shared memory and the latency of the kernel spectra between
// the barriers (stick-slip films: 46% of the shared-memory wavefronts, 40%
// issue-active, 20% DRAM).  Against the one-column pass, 40 M warp instructions
// for 64 M and 94 -> 92 us there; other sizes beside the rule (ypass_pairs).  640
// or 512 threads per SM (fewer, with more registers) measured 0-10% slower over
// 64 x 64 x 1, 355 x 145 x 3, 1024 x 256 x 2 and 1024 x 1024 x 1.
constexpr int kY2Threads = 768;  // per SM, shared out over its CTAs
template <int NZ, typename Fft>
__global__ void __launch_bounds__(kY2Threads, 1) k_ypass2(const Launch<YJob> Lc) {
  constexpr int Pin = 3 * NZ;
  extern __shared__ float4 sm4[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const YJob& J = Lc.job[j];
  const int kxa = 2 * (blockIdx.x - Lc.tile_start[j]);
  const bool has_b = kxa + 1 < J.kxh;  // an odd last column runs beside itself, stored once
  const int Q = Fft::kL ? Fft::kL : J.fy.plan.L;
  const int n_out = J.do_C ? J.n_out : 0;
  const int ch = J.ch;
  const int cb = J.do_H || ch < n_out ? Pin : 0;  // alone and at once, the coefficient planes go in place
  float4* tws = sm4 + max(Pin, cb + ch) * Q;
  int* tab = reinterpret_cast<int*>(tws + J.fy.ntw2);
  const int ny = J.ny;
  const size_t pstride = (size_t)J.kxh * ny;  // one input plane

  {
    // rows [ny, Q) are zero padding; column b follows column a
    const float2* ca = J.in + (size_t)kxa * ny;
    const int nb = has_b ? ny : 0;
    Fft::in(
        sm4, Q, Pin, J.fy, tws,
        [&](int p, int y0, int M, auto& v) {
          const float2* src = ca + p * pstride + y0;
#pragma unroll
          for (int k = 0; k < (int)(sizeof(v) / sizeof(v[0])); ++k)
            v[k] = y0 + k * M < ny ? c2_make(__ldg(src + k * M), __ldg(src + k * M + nb)) : c2_zero();
        },
        [&]() {
          for (int i = threadIdx.x; i < J.fy.ntw2; i += blockDim.x) tws[i] = __ldg(J.fy.tw2 + i);
          if (n_out)
            build_pref_table(tab, J.r + 2 * kPrefWarm + kYChunk, J.box_lo, J.box_len, J.start, Q, nullptr,
                             J.periodic != 0);
          // The kernel spectra of these columns are read after the forward FFT:
          // start moving their lines into L2 (one prefetch per 128-byte line).
          const size_t qs = (size_t)((J.kxh + 1) >> 1) * J.kyq;
          const int lines = (J.kyq + 7) / 8;  // eight quads
          const int nN = J.do_H ? 3 * NZ : 0, nT = (t_stride(NZ, true) * n_out + 1) / 2;
          for (int row = threadIdx.x / 32; row < nN + nT; row += blockDim.x / 32) {
            const float4* p = reinterpret_cast<const float4*>(row < nN ? J.Nq : J.Tq) +
                              (row < nN ? row : row - nN) * qs + (size_t)(kxa >> 1) * J.kyq;
            for (int ln = threadIdx.x % 32; ln < lines; ln += 32)
              asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 8 * ln));
          }
        });
  }
  for (int c0 = 0;; c0 += ch) {
    const int c1 = min(c0 + ch, n_out);
    const bool last = c1 >= n_out;
    const bool H = last && J.do_H;
    ypass2_mix<NZ>(J, sm4, kxa >> 1, Q, cb, c0, c1, H);
    __syncthreads();
    // inverse of the demag planes (rows y < ny straight to memory) with the
    // last coefficient planes, which follow them
    float4* first = H ? sm4 : sm4 + cb * Q;
    const int nh = H ? Pin : 0, lines = nh + c1 - c0;
    float2* oa = J.outH + (size_t)kxa * ny;
    Fft::out(first, Q, lines, J.fy, tws, [&](int p, int y0, int M, auto& v) {
      constexpr int R = (int)(sizeof(v) / sizeof(v[0]));
      if (p >= nh) {
        float4* dst = first + p * Q + y0;
#pragma unroll
        for (int k = 0; k < R; ++k) c2_store(dst + k * M, v[k]);
      } else {
        float2* dst = oa + p * pstride + y0;
#pragma unroll
        for (int k = 0; k < R; ++k)
          if (y0 + k * M < ny) {
            dst[k * M] = c2_a(v[k]);
            if (has_b) dst[k * M + ny] = c2_b(v[k]);
          }
      }
    });
    // y prefilter and the coefficient rows
    const int r = J.r, ncol = c1 - c0;
    float2* oc = J.outC + ((size_t)c0 * J.kxh + kxa) * r;
    const size_t ostride = (size_t)J.kxh * r;
    const float4* col0 = first + nh * Q;
    if (J.fir) {
      // one thread per chunk and per real or imaginary part (of both columns);
      // the two parts swap halves to store whole values
      const int nch = (r + kYChunk - 1) / kYChunk;
      const int items = 2 * ncol * nch;
      for (int base = threadIdx.x & ~31; base < items; base += blockDim.x) {
        const int at = base + (int)(threadIdx.x & 31), idx = min(at, items - 1);  // whole warps swap (items is even)
        const int o = (idx >> 1) / nch, part = idx & 1;
        const int k0 = ((idx >> 1) - o * nch) * kYChunk;
        const p2* src = reinterpret_cast<const p2*>(col0 + o * Q) + part;
        float2* dst = oc + o * ostride + part * r;
        const bool store = (part == 0 || has_b) && at < items;
        prefilter_chunk2<kYChunk>(
            k0, [&](int jj) { return src[2 * tab[jj]]; },
            [&](int k, p2 v) {
              const float2 f = p2_unpack(v);  // (column a, column b) of this part
              const float other = __shfl_xor_sync(0xffffffffu, part ? f.x : f.y, 1);
              if (store && k < r) dst[k] = part ? make_float2(other, f.y) : make_float2(f.x, other);
            });
      }
    } else {
      for (int k = threadIdx.x; ncol > 0 && k < r; k += blockDim.x) {
        const int t = tab[k + kPrefWarm];
        for (int o = 0; o < ncol; ++o) {
          const float4 v = col0[o * Q + t];
          oc[o * ostride + k] = make_float2(v.x, v.z);
          if (has_b) oc[o * ostride + k + r] = make_float2(v.y, v.w);
        }
      }
    }
    if (last) break;
    __syncthreads();  // the next planes overwrite these
  }
}

// ------------------------------------------------------------------ x inverse
__device__ __forceinline__ void xinv_put(float2* sm, int off, int Q, int kx, float2 A, float2 B) {
  // Z_k = A_k + i B_k and Z_{Q-k} = conj(A_k) + i conj(B_k), natural order; off = line start
  sm[off + kx] = make_float2(A.x - B.y, A.y + B.x);
  if (kx > 0 && 2 * kx != Q) sm[off + Q - kx] = make_float2(A.x + B.y, B.x - A.y);
}

template <unsigned RSET, int FIXP>
__global__ void __launch_bounds__(kXInvThreads, 3) k_xinv(const Launch<XInvJob> Lc) {
  extern __shared__ float2 sm[];
  pdl_wait();
  const int j = find_job(Lc.tile_start, Lc.njobs, blockIdx.x);
  const XInvJob& J = Lc.job[j];
  const int tile = blockIdx.x - Lc.tile_start[j];
  const int Q = FIXP ? FixedPlan<FIXP ? FIXP : 1>::L : J.fx.plan.L;
  const int ldl = Q + kLinePad;  // padded line stride: the lines start in different banks
  const int rpp = J.rows_per_plane;
  const int rows = J.planes * rpp;
  const int r0 = tile * kRowsPerCta;
  const int nrows = min(kRowsPerCta, rows - r0);
  const int nlines = (nrows + 1) >> 1;
  int* tab = reinterpret_cast<int*>(sm + kLines * ldl);

  // input row r of this CTA (its kx = 0 element)
  const int pa0 = r0 / rpp;
  auto rowptr = [&](int r) {
    int p = pa0, y = min(r0 + r, rows - 1) - pa0 * rpp;
    while (y >= rpp) { ++p; y -= rpp; }
    return J.in + (size_t)p * J.kxh * rpp + y;
  };
  const bool paired = (rpp & 1) == 0 && (nrows & 1) == 0;  // row pairs adjacent, 16-byte aligned
  const int n = J.kxh * nlines;
  if (paired && nlines == kLines) {
    // full tile: blockDim is a multiple of kLines, so every thread keeps one
    // line (its input row pair) for all its kx; kBatchX reads in flight (three
    // rounds of loads for a 2160-point line)
    constexpr int kBatchX = 6;
    const int l = threadIdx.x % kLines;
    const float2* src = rowptr(2 * l);
    const int step = blockDim.x / kLines;
    for (int kx0 = threadIdx.x / kLines; kx0 < J.kxh; kx0 += kBatchX * step) {
      float4 v[kBatchX];
#pragma unroll
      for (int u = 0; u < kBatchX; ++u) {
        const int kx = kx0 + u * step;
        if (kx < J.kxh) v[u] = *reinterpret_cast<const float4*>(src + (size_t)kx * rpp);
      }
#pragma unroll
      for (int u = 0; u < kBatchX; ++u) {
        const int kx = kx0 + u * step;
        if (kx < J.kxh) xinv_put(sm, l * ldl, Q, kx, make_float2(v[u].x, v[u].y), make_float2(v[u].z, v[u].w));
      }
    }
  } else if (paired) {
    // thread -> (kx, line), line fastest: a warp reads 8 runs of 64 bytes;
    // kBatchX such reads in flight per thread
    constexpr int kBatchX = 4;
    for (int base = threadIdx.x; base < n; base += kBatchX * blockDim.x) {
      float4 v[kBatchX];
#pragma unroll
      for (int u = 0; u < kBatchX; ++u) {
        const int idx = base + u * blockDim.x;
        if (idx < n) {
          const int kx = idx / nlines, l = idx - kx * nlines;
          v[u] = *reinterpret_cast<const float4*>(rowptr(2 * l) + (size_t)kx * rpp);
        }
      }
#pragma unroll
      for (int u = 0; u < kBatchX; ++u) {
        const int idx = base + u * blockDim.x;
        if (idx < n) {
          const int kx = idx / nlines, l = idx - kx * nlines;
          xinv_put(sm, l * ldl, Q, kx, make_float2(v[u].x, v[u].y), make_float2(v[u].z, v[u].w));
        }
      }
    }
  } else {
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
      const int kx = idx / nlines, l = idx - kx * nlines;
      const size_t off = (size_t)kx * rpp;
      const float2 a = rowptr(2 * l)[off];
      const float2 b = 2 * l + 1 < nrows ? rowptr(2 * l + 1)[off] : make_float2(0.f, 0.f);
      xinv_put(sm, l * ldl, Q, kx, a, b);
    }
  }
  build_pref_table(tab, J.out_len + 2 * kPrefWarm + kXChunk, J.box_lo, J.box_len, J.start, Q, J.fx.pos,
                   J.periodic != 0);
  __syncthreads();
  // natural-order input, digit-reversed output: the table above maps through it
  if constexpr (FIXP > 0)
    fft_smem_plan<kInvDif, FIXP, FixedPlan<FIXP>::L + kLinePad>(sm, nlines, J.fx.plan, J.fx.tw_f, 0, blockDim.x);
  else
    fft_smem<kInvDif, float2, RSET>(sm, ldl, nlines, J.fx.plan, J.fx.tw_f, 0, blockDim.x);

  const int r = J.out_len;
  float* out0 = J.out + (size_t)r0 * r;
  if (J.fir) {
    const int nch = (r + kXChunk - 1) / kXChunk;
    for (int idx = threadIdx.x; idx < nrows * nch; idx += blockDim.x) {
      const int rl = idx / nch;
      const int k0 = (idx - rl * nch) * kXChunk;
      const float* line = reinterpret_cast<const float*>(sm + (rl >> 1) * ldl) + (rl & 1);
      float* dst = out0 + rl * r;
      prefilter_chunk<kXChunk, float>(
          k0, r, [&](int jj) { return line[2 * tab[jj]]; }, [&](int k, float v) { dst[k] = v; });
    }
  } else {
    for (int k = threadIdx.x; k < r; k += blockDim.x) {
      const int t = 2 * tab[k + kPrefWarm];
      const float* base = reinterpret_cast<const float*>(sm) + t;
#pragma unroll
      for (int rl = 0; rl < kRowsPerCta; ++rl)
        if (rl < nrows) out0[rl * r + k] = base[(rl >> 1) * 2 * ldl + (rl & 1)];
    }
  }
}

// ------------------------------------------------------------------ host side
size_t ypass_table_bytes(int r) { return sizeof(int) * (size_t)(r + 2 * kPrefWarm + kYChunk); }

static size_t xinv_smem(int Qmax, int out_max) {
  return (size_t)kLines * (Qmax + kLinePad) * sizeof(float2) +
         sizeof(int) * (size_t)(out_max + 2 * kPrefWarm + kXChunk);
}

// the fixed plan every job's x plan is (fixed_plan_id), 0 if they differ or none is
template <typename JobT> static int x_fixed_plan(const Launch<JobT>& L) {
  int id = L.njobs > 0 ? fixed_plan_id(L.job[0].fx.plan) : 0;
  for (int i = 1; i < L.njobs; ++i)
    if (fixed_plan_id(L.job[i].fx.plan) != id) id = 0;
  return id;
}

constexpr size_t kSmemMax = 227 * 1024;              // per CTA

cudaError_t launch_xfwd(const Launch<XFwdJob>& L, int Qmax, cudaStream_t st) {
  const size_t smem =
      (size_t)kLines * (Qmax + kLinePad) * sizeof(float2) + sizeof(ushort2) * (size_t)(Qmax / 2 + 1);
  unsigned rs = 0;
  for (int i = 0; i < L.njobs; ++i) rs |= plan_radix_set(L.job[i].fx.plan);
  const int fx = x_fixed_plan(L);
  auto k = fx == 1 ? k_xfwd<kRadixSetA, 1>
           : fx == 2 ? k_xfwd<kAllRadices, 2>
           : (rs & ~kRadixSetA) == 0u ? k_xfwd<kRadixSetA, 0> : k_xfwd<kAllRadices, 0>;
  cudaError_t e = allow_smem((const void*)k, kSmemMax);
  if (e != cudaSuccess) return e;
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  return launch_chained(k, grid, kXFwdThreads, smem, st, L);
}

// The y pass of jobs of one layer count, two columns per CTA where their lines
// fit shared memory.
constexpr size_t kSmemTwo = (228 * 1024) / 2 - 1024;  // each of two CTAs on an SM

// the lengths of 64, 128, 256, 512 and 1024 cells (4 cells of margin) with their
// plans as constants.  us of whole evaluations' launches, plan at run time ->
// constant: 300 x 64 x 1 (160 points) 14.0 -> 12.5, 300 x 128 x 2 (288) 25.6 -> 24.8,
// 1024 x 256 x 2 (540) 110 -> 94, 450 x 512 x 1 (1080) 79 -> 64 and x 3 213 -> 198,
// 1024 x 1024 x 1 (2160) 328 -> 300
using YPairPlans =
    PairPlans<CtPair<4, 8, 5>, CtPair<4, 8, 9>, CtPair<12, 9, 5>, CtPair<10, 12, 9>, CtPair<6, 8, 9, 5>>;
template <int NZ> struct YPass2 {
  // three layers: short lines, and 1080 points (ypass_pairs)
  static constexpr bool takes(int L) { return pairs_fit(NZ, L) && (NZ < 3 || L <= 360 || L > 640); }
  template <typename Fft> static auto build() { return &k_ypass2<NZ, Fft>; }
};
bool ypass_plan_compiled(const FftPlanDev& P) { return YPairPlans::has(P); }

// Whether a source of kxh columns takes two per CTA.  `both`: demag and
// coefficient planes at once, in a whole evaluation, whose launch takes both
// films; else planes of one kind of one film.
//
// Pairs halve the CTAs and double their shared memory, so they pay where the
// columns are many against the 152 SMs (one column per CTA: three CTAs a SM up to
// two layers, two at three) and their lines few and short enough to be taken at
// once; compiled plans pay further.  The lines are drawn where neither form is
// slower, from 1200 sizes (20 to 1000 cells in x, 20 to 1024 in y, one to three
// layers, the three kinds of call).  us of the pass, one column -> two:
//   short lines: whole evaluations of 300 x 64 x 1 (160 points) 23.5 -> 12.7, 300 x 100 x
//     3 (240) 34.4 -> 28.5, 145 x 100 x 3 (322 columns) 24.7 -> 23.4, but x 2 16.1 -> 18.1;
//     40 x 64 x 1 (compiled, few columns) 14.4 -> 10.3, 40 x 100 x 3 (not) 14.4 -> 20.7;
//   up to 640 points: 600 x 300 x 1 66.6 -> 60.9, 145 x 256 x 1 19.2 -> 20.8; stray field
//     calls of 450 x 300 x 1 34.8 -> 21.7, x 2 39.1 -> 28.3;
//   long lines: 600 x 1024 x 1 (2160, compiled) 248 -> 189 whole, 73 -> 82 the stray
//     field alone; 600 x 400 x 2 (864, planes in five chunks) 130 -> 178.
constexpr int kSMs = 152;
bool ypass_pairs(int nz, int Qy, int kxh, bool both) {
  if (!pairs_fit(nz, Qy)) return false;
  const bool compiled = YPairPlans::has_length(Qy);
  const int cols = both ? 2 * kxh : kxh;
  if (Qy <= 360)
    return kxh >= 2 * kSMs || (both && nz != 2 && kxh >= kSMs) || (compiled && nz * Qy <= 320);
  if (nz == 1 && Qy <= 750 && cols >= (Qy > 640 ? 6 : both ? 4 : 3) * kSMs) return true;
  if (nz == 2 && Qy <= 640 && !both && kxh >= 3 * kSMs && kxh < 6 * kSMs) return true;
  return compiled && both && (Qy > 640 ? cols >= 6 * kSMs : nz == 2 && cols >= 10 * kSMs);
}

static size_t ypass2_smem(const YJob& J, int ch) {
  const int n_out = J.do_C ? J.n_out : 0;
  const int cb = J.do_H || ch < n_out ? 3 * J.nz : 0;
  return ((size_t)max(3 * J.nz, cb + ch) * J.fy.plan.L + J.fy.ntw2) * sizeof(float4) +
         ypass_table_bytes(n_out ? J.r : 0);
}

// Coefficient planes at a time: all of them, or the most that let two CTAs
// share an SM, or the most that fit (pairs_fit: two at least).  Chunks start on
// whole quads of the kernel spectra: one layer's hold two planes.
static int ypass2_chunk(const YJob& J) {
  const int n_out = J.do_C ? J.n_out : 0;
  for (size_t limit : {kSmemTwo, kSmemMax}) {
    if (ypass2_smem(J, n_out) <= limit) return max(n_out, 1);
    for (int ch = n_out - 1; ch >= 1; --ch)
      if (ypass2_smem(J, ch) <= limit && (J.nz > 1 || ch % 2 == 0)) return ch;
  }
  return 0;
}

// The jobs of one layer count, two columns per CTA.
template <int NZ> static cudaError_t launch_ypass_pairs(const Launch<YJob>& L0, cudaStream_t st) {
  Launch<YJob> L = L0;
  int tiles = 0;
  size_t smem = 0;
  for (int i = 0; i < L.njobs; ++i) {
    YJob& J = L.job[i];
    J.ch = ypass2_chunk(J);
    if (J.ch == 0) return cudaErrorInvalidConfiguration;
    smem = max(smem, ypass2_smem(J, J.ch));
    L.tile_start[i] = tiles;
    tiles += (J.kxh + 1) / 2;
  }
  L.tile_start[L.njobs] = tiles;
  auto k = YPairPlans::kernel<YPass2<NZ>>(L, &YJob::fy);
  cudaError_t e = allow_smem((const void*)k, kSmemMax);
  if (e != cudaSuccess || tiles == 0) return e;
  const int ctas = min(3, max(1, (int)(228 * 1024 / (smem + 1024))));
  return launch_chained(k, tiles, kY2Threads / ctas / 32 * 32, smem, st, L);
}

// ... and one column per CTA.
template <int NZ> static cudaError_t launch_ypass_columns(const Launch<YJob>& L, size_t smem, cudaStream_t st) {
  unsigned rs = 0;
  bool fix540 = true;
  for (int i = 0; i < L.njobs; ++i) {
    rs |= plan_radix_set(L.job[i].fy.plan);
    fix540 = fix540 && fixed_plan_id(L.job[i].fy.plan) == 3;
  }
  auto k = fix540 ? k_ypass<NZ, kRadixSetA, true>
                  : (rs & ~kRadixSetA) == 0u ? k_ypass<NZ, kRadixSetA, false> : k_ypass<NZ, kAllRadices, false>;
  cudaError_t e = allow_smem((const void*)k, kSmemMax);
  if (e != cudaSuccess || L.tile_start[L.njobs] == 0) return e;
  return launch_chained(k, L.tile_start[L.njobs], kYThreads, smem, st, L);
}

// Jobs of different layer counts, or of one and two columns per CTA, go to
// separate launches of the matching kernel.
cudaError_t launch_ypass(const Launch<YJob>& L, size_t smem, cudaStream_t st) {
  for (int nz = 1; nz <= kMaxNz; ++nz)
    for (int pairs = 0; pairs < 2; ++pairs) {
      Launch<YJob> S{};
      int tiles = 0;
      for (int i = 0; i < L.njobs; ++i) {
        if (L.job[i].nz != nz || L.job[i].pairs != pairs) continue;
        S.job[S.njobs] = L.job[i];
        S.tile_start[S.njobs] = tiles;
        tiles += L.job[i].kxh;
        ++S.njobs;
      }
      if (S.njobs == 0) continue;
      S.tile_start[S.njobs] = tiles;
      cudaError_t e = pairs ? (nz == 1   ? launch_ypass_pairs<1>(S, st)
                               : nz == 2 ? launch_ypass_pairs<2>(S, st)
                                         : launch_ypass_pairs<3>(S, st))
                      : nz == 1 ? launch_ypass_columns<1>(S, smem, st)
                      : nz == 2 ? launch_ypass_columns<2>(S, smem, st)
                      : nz == 3 ? launch_ypass_columns<3>(S, smem, st)
                                : launch_ypass_columns<4>(S, smem, st);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

cudaError_t launch_xinv(const Launch<XInvJob>& L, int Qmax, cudaStream_t st) {
  int out_max = 0;
  for (int i = 0; i < L.njobs; ++i) out_max = max(out_max, L.job[i].out_len);
  const size_t smem = xinv_smem(Qmax, out_max);
  unsigned rs = 0;
  for (int i = 0; i < L.njobs; ++i) rs |= plan_radix_set(L.job[i].fx.plan);
  const int fx = x_fixed_plan(L);
  auto k = fx == 1 ? k_xinv<kRadixSetA, 1>
           : fx == 2 ? k_xinv<kAllRadices, 2>
           : (rs & ~kRadixSetA) == 0u ? k_xinv<kRadixSetA, 0> : k_xinv<kAllRadices, 0>;
  cudaError_t e = allow_smem((const void*)k, kSmemMax);
  if (e != cudaSuccess) return e;
  const int grid = L.tile_start[L.njobs];
  if (grid == 0) return cudaSuccess;
  return launch_chained(k, grid, kXInvThreads, smem, st, L);
}

}  // namespace mm
