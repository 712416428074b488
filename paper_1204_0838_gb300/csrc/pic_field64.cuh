// pic_field64.cuh -- the FP64 field update (Eq. perfDispMaxwell) with its
// differences and smoothing in 64-bit fixed point on the integer pipes.
//
// What bounded the FP64 kernels that these replace: the FP64 pipe, 77-83 % busy
// (about 110 FP64 instructions per cell and step; this GPU retires 0.5 T/s of
// them).  Here a CTA stages a 4x8x32 block of a field with its halo, converts it
// to int64 at a power of two per block and component with max|F| 2^s < 2^60, and
// forms differences, the smoothing's sums and the products with constant
// weights as integers (pic_fixed64.cuh); 6 FP64 instructions per cell and kernel
// are left, which add the increments to the stored fields.
//
// Measured: step of a vacuum box of 8.4 M cells 2.00 -> 0.87 ms (magnetic kernel
// 1.6 -> 0.47, electric kernel 0.45 -> 0.30; the 12 values read and written per
// cell and kernel are 0.24 ms at the copy rate); 118 M particle step on 101 M cells
// 93 -> 80 ms.  About 560 (electric) and 990 (magnetic) instructions per 32 cells,
// issued 40-45 % of the time, bound both; half of them convert between doubles
// and integers.
//
// The increments carry an absolute error of a few units of 2^-59 of the block's
// largest value, below the 2^-53 rounding of that value itself; each component
// of a curl takes the coarser scale of the two components that enter it.  A
// block that holds a NaN or an infinity takes the FP64 arithmetic instead, cell
// by cell, so that non-finite values spread as they do in FP64.
#pragma once

#include "pic_fixed64.cuh"
#include "pic_kernels.cuh"

namespace pic {

// Constant weights, split: smoothing centre, two edges, corner per axis at 2^62;
// dt/2 / d at 2^63 and dt / d at 2^62 per axis.
struct FieldConst64 {
  S32 s[3][4];
  S32 hd[3], fd[3];
  double idt, ihdt;  // 1 / dt, 2 / dt
};

// Largest exponent of the block's values, per component (sh: 3 shared ints,
// zero on entry; barriers inside).  Returns false if a value is not finite.
__device__ __forceinline__ bool block_scales(const int (&emax)[3], int* sh, int (&e)[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)emax[c]);
    if ((threadIdx.x & 31) == 0) atomicMax(sh + c, (int)m);
  }
  __syncthreads();
  bool finite = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    finite = finite && sh[c] != 0x7FF;
    e[c] = max(sh[c], kFieldMinExp);
  }
  return finite;
}

// x w / 2^63 (one product), one bit more than x w / 2^64.
__device__ __forceinline__ long long scaled(long long x, S32 w) {
  Acc32 a = {0LL, kRound2};
  acc32(a, split32(x), w);
  return acc32_result2(a);
}

// a - b for a at scale sa, b at sb, at the coarser of the two; the finer one is
// rounded to nearest (cut off, it would give the increments of a block a mean error
// of half a unit that recurs every step).  |a|, |b| < 2^61.
__device__ __forceinline__ long long coarser(long long a, int sh) {
  const int r = min(sh, 62);
  return (a + ((1LL << r) >> 1)) >> r;
}
__device__ __forceinline__ long long aligned_diff(long long a, int sa, long long b, int sb) {
  const int s = min(sa, sb);
  return coarser(a, sa - s) - coarser(b, sb - s);
}

// E^{n+1} = E^n + dt (curl B^{n+1/2} - J); hb holds B^{n+1/2}.
constexpr int EB_N = (CB_X + 1) * (CB_Y + 1) * (CB_Z + 1);
__global__ void __launch_bounds__(256, 2)
    k_e_update64(Geom<double> g, Fields<double> f, Fields<double> hb, FieldCoef<double> fc, FieldConst64 k64,
                 Pml<double> pm) {
  if (!dyn_prologue(g)) return;
  __shared__ long long sB[3][EB_N];  // origin (bx-1, by-1, bz-1)
  __shared__ int sh[3];
  const int bx = blockIdx.x * CB_X, by = blockIdx.y * CB_Y, bz = blockIdx.z * CB_Z;
  const int tid = threadIdx.x;
  constexpr int kIt = (EB_N + 255) / 256, kPer = CB_X * CB_Y * CB_Z / 256;
  constexpr int NY = CB_Y + 1, NZ = CB_Z + 1;
  if (tid < 3) sh[tid] = 0;
  long long raw[kIt][3];
  int emax[3] = {0, 0, 0};
#pragma unroll
  for (int t = 0; t < kIt; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % NZ, r = q / NZ, ly = r % NY, lx = r / NY;
    int s = q < EB_N ? slab_of(g, bx - 1 + lx) : -1;
    int j = by - 1 + ly, k = bz - 1 + lz;
    if (g.pml) {
      if (j < 0 || j >= g.ny || k < 0 || k >= g.nz) s = -1;
    } else {
      j = j < 0 ? j + g.ny : (j >= g.ny ? -1 : j);  // cells beyond the far end are not read
      k = k < 0 ? k + g.nz : (k >= g.nz ? -1 : k);
      if (j < 0 || k < 0) s = -1;
    }
    const size_t gi = s < 0 ? 0 : (size_t)s * g.nyz + (size_t)j * g.nz + k;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      raw[t][c] = s < 0 ? 0LL : __double_as_longlong(hb.c[c][gi]);
      emax[c] = max(emax[c], (int)((unsigned long long)raw[t][c] >> 52) & 0x7FF);
    }
  }
  // E and J of the thread's cells, in flight with the staged values
  double pe[kPer][3], pj[kPer][3];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % CB_Z, r = q / CB_Z;
    const int i = bx + r / CB_Y, j = by + r % CB_Y, k = bz + lz;
    const bool in = i < g.nx && j < g.ny && k < g.nz;
    const size_t id = in ? (size_t)slab_of(g, i) * g.nyz + (size_t)j * g.nz + k : 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      pe[t][c] = f.c[EX + c][id];
      pj[t][c] = f.c[JX + c][id];
    }
  }
  __syncthreads();
  int e[3];
  const bool finite = block_scales(emax, sh, e);
  if (!finite) {  // uniform over the block
    for (int t = 0; t < kPer; ++t) {
      const int q = tid + 256 * t;
      const int lz = q % CB_Z, r = q / CB_Z;
      const int i = bx + r / CB_Y, j = by + r % CB_Y, k = bz + lz;
      if (i < g.nx && j < g.ny && k < g.nz) e_update_cell(g, f, hb, fc, pm, i, j, k);
    }
    return;
  }
#pragma unroll
  for (int t = 0; t < kIt; ++t) {
    const int q = tid + 256 * t;
    if (q < EB_N)
#pragma unroll
      for (int c = 0; c < 3; ++c) sB[c][q] = field_fixed(raw[t][c], e[c]);
  }
  __syncthreads();
  int sc[3];  // scale of the products
#pragma unroll
  for (int c = 0; c < 3; ++c) sc[c] = kFieldBits - 2 + 1023 - e[c];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % CB_Z, r = q / CB_Z, ly = r % CB_Y, lx = r / CB_Y;
    const int i = bx + lx, j = by + ly, k = bz + lz;
    if (i >= g.nx || j >= g.ny || k >= g.nz) continue;
    const int slab = slab_of(g, i);
    const size_t id = (size_t)slab * g.nyz + (size_t)j * g.nz + k;
    const int p = ((lx + 1) * NY + ly + 1) * NZ + lz + 1;
    const long long vx = sB[0][p], vy = sB[1][p], vz = sB[2][p];
    const long long yBz = scaled(vz - sB[2][p - NZ], k64.fd[1]), zBy = scaled(vy - sB[1][p - 1], k64.fd[2]);
    const long long zBx = scaled(vx - sB[0][p - 1], k64.fd[2]), xBz = scaled(vz - sB[2][p - NY * NZ], k64.fd[0]);
    const long long xBy = scaled(vy - sB[1][p - NY * NZ], k64.fd[0]), yBx = scaled(vx - sB[0][p - NZ], k64.fd[1]);
    double dE[3];
    const int jr = pm.L ? pml_row(j, g.ny, pm.L) : -1, kr = pm.L ? pml_row(k, g.nz, pm.L) : -1;
    if (jr >= 0 || kr >= 0) {  // memory variables (times dt): y and z at nodes
      double dyBz = fixed_to_double(yBz, sc[2]), dzBy = fixed_to_double(zBy, sc[1]);
      double dzBx = fixed_to_double(zBx, sc[0]), dyBx = fixed_to_double(yBx, sc[0]);
      if (jr >= 0) {
        const double a = pm.cy[j] * k64.idt, b = pm.cy[g.ny + j];
        const size_t pi = ((size_t)slab * pm.rows + jr) * g.nz + k;
        const double p0 = b * pm.py[0][pi] + a * dyBz, p1 = b * pm.py[1][pi] + a * dyBx;
        pm.py[0][pi] = p0;
        pm.py[1][pi] = p1;
        dyBz += fc.dt * p0;
        dyBx += fc.dt * p1;
      }
      if (kr >= 0) {
        const double a = pm.cz[k] * k64.idt, b = pm.cz[g.nz + k];
        const size_t pi = ((size_t)slab * g.ny + j) * pm.rows + kr;
        const double p0 = b * pm.pz[0][pi] + a * dzBy, p1 = b * pm.pz[1][pi] + a * dzBx;
        pm.pz[0][pi] = p0;
        pm.pz[1][pi] = p1;
        dzBy += fc.dt * p0;
        dzBx += fc.dt * p1;
      }
      dE[0] = dyBz - dzBy;
      dE[1] = dzBx - fixed_to_double(xBz, sc[2]);
      dE[2] = fixed_to_double(xBy, sc[1]) - dyBx;
    } else {
      dE[0] = fixed_to_double(aligned_diff(yBz, sc[2], zBy, sc[1]), min(sc[2], sc[1]));
      dE[1] = fixed_to_double(aligned_diff(zBx, sc[0], xBz, sc[2]), min(sc[0], sc[2]));
      dE[2] = fixed_to_double(aligned_diff(xBy, sc[1], yBx, sc[0]), min(sc[1], sc[0]));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) f.c[EX + c][id] = pe[t][c] + fma(-fc.dt, pj[t][c], dE[c]);
  }
}

// Smoothed curl and the magnetic half steps, as k_curl_tiled.
constexpr size_t kCurl64Smem = 8 * (3 * (size_t)CE_N + 2 * (size_t)(SXN + SYN + SZN));
__global__ void __launch_bounds__(256, 2)
    k_curl64(Geom<double> g, Smooth<double> S, Fields<double> f, Fields<double> hb, FieldCoef<double> fc,
             FieldConst64 k64, int mode, FieldSpan sp, Pml<double> pm) {
  if (!dyn_prologue(g)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sh[3];
  long long* sE = reinterpret_cast<long long*>(smem_raw);  // [3][CE_X][CE_Y][CE_Z], origin (bx-1, by-1, bz-1)
  long long* sSxEy = sE + 3 * CE_N;                        // [CB_X+1][CB_Y][CB_Z]
  long long* sSxEz = sSxEy + SXN;
  long long* sSyEz = sSxEz + SXN;                          // [CB_X][CB_Y+1][CB_Z]
  long long* sSyEx = sSyEz + SYN;
  long long* sSzEx = sSyEx + SYN;                          // [CB_X][CB_Y][CB_Z+1]
  long long* sSzEy = sSzEx + SZN;
  const int bx = blockIdx.x * sp.step, bx1 = min(bx + sp.width, g.nx), by = blockIdx.y * CB_Y, bz = blockIdx.z * CB_Z;
  const int tid = threadIdx.x;
  constexpr int kPer = CB_X * CB_Y * CB_Z / 256;
  int e[3];
  bool finite;
  double pb[kPer][3];  // H (mode 1) or B (mode 0) of the thread's cells
  if (tid < 3) sh[tid] = 0;
  {
    constexpr int kIt = (CE_N + 255) / 256;
    long long raw[kIt][3];
    int emax[3] = {0, 0, 0};
#pragma unroll
    for (int t = 0; t < kIt; ++t) {
      const int q = tid + 256 * t;
      const int lz = q % CE_Z, r = q / CE_Z, ly = r % CE_Y, lx = r / CE_Y;
      int s = q < CE_N ? slab_of(g, bx - 1 + lx) : -1;
      int j = by - 1 + ly, k = bz - 1 + lz;
      if (g.pml) {  // zero beyond the grid
        if (j < 0 || j >= g.ny || k < 0 || k >= g.nz) s = -1;
      } else {      // periodic; a block may exceed a small ny or nz more than once
        j = j < 0 ? j + g.ny : (j >= g.ny ? j - g.ny : j);
        k = k < 0 ? k + g.nz : (k >= g.nz ? k - g.nz : k);
        if ((unsigned)j >= (unsigned)g.ny) j = wrapi(j, g.ny);
        if ((unsigned)k >= (unsigned)g.nz) k = wrapi(k, g.nz);
      }
      const size_t gi = s < 0 ? 0 : (size_t)s * g.nyz + (size_t)j * g.nz + k;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        raw[t][c] = s < 0 ? 0LL : __double_as_longlong(f.c[EX + c][gi]);
        emax[c] = max(emax[c], (int)((unsigned long long)raw[t][c] >> 52) & 0x7FF);
      }
    }
#pragma unroll
    for (int t = 0; t < kPer; ++t) {  // in flight with the staged values
      const int q = tid + 256 * t;
      const int lz = q % CB_Z, r = q / CB_Z;
      const int i = bx + r / CB_Y, j = by + r % CB_Y, k = bz + lz;
      const bool in = i < bx1 && j < g.ny && k < g.nz;
      const size_t id = in ? (size_t)slab_of(g, i) * g.nyz + (size_t)j * g.nz + k : 0;
#pragma unroll
      for (int c = 0; c < 3; ++c) pb[t][c] = mode == 1 ? hb.c[c][id] : f.c[BX + c][id];
    }
    __syncthreads();
    finite = block_scales(emax, sh, e);
    if (finite)
#pragma unroll
      for (int t = 0; t < kIt; ++t) {
        const int q = tid + 256 * t;
        if (q < CE_N)
#pragma unroll
          for (int c = 0; c < 3; ++c) sE[c * CE_N + q] = field_fixed(raw[t][c], e[c]);
      }
  }
  if (!finite) {  // uniform over the block
    for (int t = 0; t < kPer; ++t) {
      const int q = tid + 256 * t;
      const int lz = q % CB_Z, r = q / CB_Z;
      const int i = bx + r / CB_Y, j = by + r % CB_Y, k = bz + lz;
      if (i < bx1 && j < g.ny && k < g.nz) curl_cell(g, S, f, hb, fc, pm, mode, i, j, k);
    }
    return;
  }
  __syncthreads();
  {
    auto E = [&](int c, int p) -> long long { return sE[c * CE_N + p]; };
    // sum over the 3x3 points around p with steps a, b: at 2^(s - 1)
    auto smooth = [&](int c, int p, int a, int b, const S32(&w)[4]) -> long long {
      const long long e1 = E(c, p + a) + E(c, p - a), e2 = E(c, p + b) + E(c, p - b);
      const long long cr = (E(c, p + a + b) + E(c, p + a - b)) + (E(c, p - a + b) + E(c, p - a - b));
      Acc32 s = {0LL, kRound2};
      acc32(s, split32(E(c, p)), w[0]);
      acc32(s, split32(e1), w[1]);
      acc32(s, split32(e2), w[2]);
      acc32(s, split32(cr), w[3]);
      return acc32_result2(s);
    };
    constexpr int PX = CE_Y * CE_Z, PY = CE_Z;
    for (int q = tid; q < SXN; q += 256) {
      const int lz = q % CB_Z, r = q / CB_Z;
      const int p = (r / CB_Y + 1) * PX + (r % CB_Y + 1) * PY + lz + 1;
      sSxEy[q] = smooth(1, p, PY, 1, k64.s[0]);
      sSxEz[q] = smooth(2, p, PY, 1, k64.s[0]);
    }
    for (int q = tid; q < SYN; q += 256) {
      const int lz = q % CB_Z, r = q / CB_Z;
      const int p = (r / (CB_Y + 1) + 1) * PX + (r % (CB_Y + 1) + 1) * PY + lz + 1;
      sSyEz[q] = smooth(2, p, PX, 1, k64.s[1]);
      sSyEx[q] = smooth(0, p, PX, 1, k64.s[1]);
    }
    for (int q = tid; q < SZN; q += 256) {
      const int lz = q % (CB_Z + 1), r = q / (CB_Z + 1);
      const int p = (r / CB_Y + 1) * PX + (r % CB_Y + 1) * PY + lz + 1;
      sSzEx[q] = smooth(0, p, PX, PY, k64.s[2]);
      sSzEy[q] = smooth(1, p, PX, PY, k64.s[2]);
    }
  }
  __syncthreads();
  int sc[3];  // scale of the products
#pragma unroll
  for (int c = 0; c < 3; ++c) sc[c] = kFieldBits - 2 + 1023 - e[c];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % CB_Z, r = q / CB_Z, ly = r % CB_Y, lx = r / CB_Y;
    const int i = bx + lx, j = by + ly, k = bz + lz;
    if (i >= bx1 || j >= g.ny || k >= g.nz) continue;
    const int x0 = (lx * CB_Y + ly) * CB_Z + lz, x1 = x0 + CB_Y * CB_Z;
    const int y0 = (lx * (CB_Y + 1) + ly) * CB_Z + lz, y1 = y0 + CB_Z;
    const int z0 = (lx * CB_Y + ly) * (CB_Z + 1) + lz;
    const int slab = slab_of(g, i);
    const size_t id = (size_t)slab * g.nyz + (size_t)j * g.nz + k;
    // dt/2 times D_y S_y Ez, D_z S_z Ey; D_z S_z Ex, D_x S_x Ez; D_x S_x Ey, D_y S_y Ex
    const long long yEz = scaled(sSyEz[y1] - sSyEz[y0], k64.hd[1]), zEy = scaled(sSzEy[z0 + 1] - sSzEy[z0], k64.hd[2]);
    const long long zEx = scaled(sSzEx[z0 + 1] - sSzEx[z0], k64.hd[2]), xEz = scaled(sSxEz[x1] - sSxEz[x0], k64.hd[0]);
    const long long xEy = scaled(sSxEy[x1] - sSxEy[x0], k64.hd[0]), yEx = scaled(sSyEx[y1] - sSyEx[y0], k64.hd[1]);
    double dB[3];
    const int jr = pm.L ? pml_row(j, g.ny, pm.L) : -1, kr = pm.L ? pml_row(k, g.nz, pm.L) : -1;
    if (jr >= 0 || kr >= 0) {  // memory variables: y and z at half nodes
      CurlD<double> d;
      d.dyEz = fixed_to_double(yEz, sc[2]) * k64.ihdt;
      d.dzEy = fixed_to_double(zEy, sc[1]) * k64.ihdt;
      d.dzEx = fixed_to_double(zEx, sc[0]) * k64.ihdt;
      d.dxEz = fixed_to_double(xEz, sc[2]) * k64.ihdt;
      d.dxEy = fixed_to_double(xEy, sc[1]) * k64.ihdt;
      d.dyEx = fixed_to_double(yEx, sc[0]) * k64.ihdt;
      curl_layers(g, pm, mode, slab, j, k, d);
      dB[0] = fc.hdt * (d.dyEz - d.dzEy);
      dB[1] = fc.hdt * (d.dzEx - d.dxEz);
      dB[2] = fc.hdt * (d.dxEy - d.dyEx);
    } else {
      dB[0] = fixed_to_double(aligned_diff(yEz, sc[2], zEy, sc[1]), min(sc[2], sc[1]));
      dB[1] = fixed_to_double(aligned_diff(zEx, sc[0], xEz, sc[2]), min(sc[0], sc[2]));
      dB[2] = fixed_to_double(aligned_diff(xEy, sc[1], yEx, sc[0]), min(sc[1], sc[0]));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (mode == 1) {
        const double b = pb[t][c] - dB[c];
        f.c[BX + c][id] = b;
        hb.c[c][id] = b - dB[c];
      } else {
        hb.c[c][id] = pb[t][c] - dB[c];
      }
    }
  }
}

}  // namespace pic
