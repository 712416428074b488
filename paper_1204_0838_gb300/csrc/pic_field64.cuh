// pic_field64.cuh -- the FP64 field update (Eq. perfDispMaxwell) with its
// differences and smoothing in 64-bit fixed point on the integer pipes.
//
// What bounded the FP64 kernels that these replace: the FP64 pipe, 77-83 % busy
// (about 110 FP64 instructions per cell and step; this GPU retires 0.5 T/s of
// them).  Here a CTA stages an 8x8x16 block of a field with its halo, converts it
// to int64 at a power of two per block and component with max|F| 2^s < 2^60, and
// forms differences, the smoothing's sums and the products with constant
// weights as integers (pic_fixed64.cuh); 6 FP64 instructions per cell and kernel
// are left, which add the increments to the stored fields.
//
// An increment's error is 2^-60 to 2^-61 of the block's largest value (rms).  Where
// that is more than FP64 arithmetic would make of the values at hand, the derivative
// is formed in FP64 (WeakTest): 0.7 % of them in a laser pulse in vacuum, 4 % around a
// tightly focused one in plasma.  Each component of a curl takes the coarser scale of
// the two that enter it.  A block that holds a NaN, an infinity or a value above 2^1021
// takes FP64 arithmetic as a whole, so that non-finite values spread as they do in
// FP64; so does, in the magnetic kernel, one that is mostly weak.
//
// Measured, FP64 arithmetic -> here: step of a vacuum box of 8.4 M cells 2.00 -> 1.03 ms
// (magnetic kernel 1.6 -> 0.60, electric kernel 0.45 -> 0.35; the 12 values read and
// written per cell and kernel are 0.24 ms at the copy rate).  Without the test and what
// it sends to FP64 the two kernels took 0.47 and 0.30 ms.
#pragma once

#include "pic_fixed64.cuh"
#include "pic_kernels.cuh"

namespace pic {

// A block of cells, with the staged fields one cell beyond it, and the points of the
// smoothed fields S_x Ey, S_x Ez; S_y Ez, S_y Ex; S_z Ex, S_z Ey.  Compact, for one
// scale to serve it: along z above all, where a pulse falls off.  (4x8x32 blocks, with
// products two bits coarser and the test's bounds accordingly: four to six times as many
// derivatives in FP64, vacuum step 1.44 ms instead of 1.09.)
constexpr int FB_X = 8, FB_Y = 8, FB_Z = 16;
constexpr int FE_X = FB_X + 2, FE_Y = FB_Y + 2, FE_Z = FB_Z + 2;
constexpr int FE_N = FE_X * FE_Y * FE_Z;
constexpr int FXN = (FB_X + 1) * FB_Y * FB_Z, FYN = FB_X * (FB_Y + 1) * FB_Z, FZN = FB_X * FB_Y * (FB_Z + 1);
static_assert(FB_Z == 16 && FB_Y % 2 == 0, "a warp: two rows of 16 cells in one x slab");

// Constant weights, split: smoothing centre, two edges, corner per axis at 2^62, and
// the upper 15 bits of their low words; dt/2 / d at 2^63 and dt / d at 2^62 per axis.
struct FieldConst64 {
  S32 s[3][4];
  int s17[3][4];
  S32 hd[3], fd[3];
  double idt, ihdt;  // 1 / dt, 2 / dt
};

// High word of a double's magnitude: its exponent and leading bits.
__device__ __forceinline__ int high_bits(long long b) { return (int)((unsigned long long)b >> 32) & 0x7FFFFFFF; }
__device__ __forceinline__ int high_bits(double v) { return __double2hiint(v) & 0x7FFFFFFF; }

// Largest exponent of the block's values per component, from the largest high words
// (sh: 3 shared ints, zero on entry; barriers inside).  Returns false if a value is
// not finite, or so large that a sum may not be.
__device__ __forceinline__ bool block_scales(const int (&hmax)[3], int* sh, int (&e)[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)hmax[c]);
    if ((threadIdx.x & 31) == 0) atomicMax(sh + c, (int)m);
  }
  __syncthreads();
  bool finite = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    finite = finite && sh[c] < 0x7FC00000;
    e[c] = max(sh[c] >> 20, kFieldMinExp);
  }
  return finite;
}

// The six derivatives of a curl, in the order of CurlD, are of the components z, y, x,
// z, y, x; two by two they enter the components x, y, z of the curl.  One that takes
// part from values far below the block's largest keeps its precision only in FP64.
// It is strong if one of its operands, at the cell or up to two cells to either side
// along z, comes within a bound of the largest value M of its component, or if the
// value that takes the increment does.  The bounds lie where the error in fixed point
// is that of FP64 in the operands or in the sum (2^-54.3 of it, rms):
//   magnetic: 2^-61.4 M against 2^-54 of the smoothed operands; 2^-8 to 2^-7 of M, and
//   2^-7 to 2^-6 for the sum;
//   electric: 2^-60.2 M against the 2^-53.8 that the operands carry; 2^-7 to 2^-6 both.
// All lanes of a warp, two rows of cells, call.
struct WeakTest {
  unsigned window;
  int least;      // high word from which an operand is strong
  int target[3];  // high word from which the sum is strong, per differentiated component
  __device__ __forceinline__ WeakTest(const int (&e)[3], const int* sh, int least_bit) : least(1 << (least_bit - 32)) {
    const int lane = threadIdx.x & 15;
    window = ((0x1Fu << lane >> 2) & 0xFFFFu) << (threadIdx.x & 16);
#pragma unroll
    for (int c = 0; c < 3; ++c) target[c] = sh[c] == 0 ? -1 : (e[c] - 6) << 20;  // an all-zero component is exact
  }
  // bit n if derivative n, with operands x and y, is weak; hi: high word of the value
  // that takes the increment (-1: not to be looked at)
  __device__ __forceinline__ unsigned operator()(int n, long long x, long long y, int hi) const {
    const int a = (int)(x >> 32), b = (int)(y >> 32);
    const bool near = __ballot_sync(0xffffffffu, ((a ^ (a >> 31)) | (b ^ (b >> 31))) >= least) & window;
    return !near && hi < target[2 - n % 3] ? 1u << n : 0u;
  }
};

// x w / 2^(64 - K) (one product).
template <int K>
__device__ __forceinline__ long long scaled(long long x, S32 w) {
  Acc32 a = {0LL, 1LL << (31 - K)};
  acc32(a, split32(x), w);
  return (a.H << K) + (a.M >> (32 - K));
}

// a - b for a at scale sa, b at sb, at the coarser of the two; the finer one is
// rounded to nearest (cut off, it would give the increments of a block a mean error
// of half a unit that recurs every step).  |a|, |b| <= 2^61.
__device__ __forceinline__ long long coarser(long long a, int sh) {
  const int r = min(sh, 62);
  return (a + ((1LL << r) >> 1)) >> r;
}
__device__ __forceinline__ long long aligned_diff(long long a, int sa, long long b, int sb) {
  const int s = min(sa, sb);
  return coarser(a, sa - s) - coarser(b, sb - s);
}

// E^{n+1} = E^n + dt (curl B^{n+1/2} - J); hb holds B^{n+1/2}.
constexpr int EB_N = (FB_X + 1) * (FB_Y + 1) * (FB_Z + 1);
__global__ void __launch_bounds__(256, 2)
    k_e_update64(Geom<double> g, Fields<double> f, Fields<double> hb, FieldCoef<double> fc, FieldConst64 k64,
                 Pml<double> pm) {
  if (!dyn_prologue(g)) return;
  __shared__ long long sB[3][EB_N];  // origin (bx-1, by-1, bz-1)
  __shared__ int sh[3];
  const int bx = blockIdx.z * FB_X, by = blockIdx.y * FB_Y, bz = blockIdx.x * FB_Z;
  const int tid = threadIdx.x;
  constexpr int kIt = (EB_N + 255) / 256, kPer = FB_X * FB_Y * FB_Z / 256;
  constexpr int NY = FB_Y + 1, NZ = FB_Z + 1;
  if (tid < 3) sh[tid] = 0;
  long long raw[kIt][3];
  int hmax[3] = {0, 0, 0};
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
      hmax[c] = max(hmax[c], high_bits(raw[t][c]));
    }
  }
  // E and J of the thread's cells, in flight with the staged values
  double pe[kPer][3], pj[kPer][3];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % FB_Z, r = q / FB_Z;
    const int i = bx + r / FB_Y, j = by + r % FB_Y, k = bz + lz;
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
  const bool finite = block_scales(hmax, sh, e);
  if (!finite) {  // uniform over the block
    for (int t = 0; t < kPer; ++t) {
      const int q = tid + 256 * t;
      const int lz = q % FB_Z, r = q / FB_Z;
      const int i = bx + r / FB_Y, j = by + r % FB_Y, k = bz + lz;
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
  const WeakTest weak_test(e, sh, kFieldBits - 7);
  int sc[3];  // scale of the products
#pragma unroll
  for (int c = 0; c < 3; ++c) sc[c] = kFieldBits - 1 + 1023 - e[c];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % FB_Z, r = q / FB_Z, ly = r % FB_Y, lx = r / FB_Y;
    const int i = bx + lx, j = by + ly, k = bz + lz;
    if (i >= g.nx) continue;  // uniform over a warp
    const int slab = slab_of(g, i);
    const size_t id = (size_t)slab * g.nyz + (size_t)j * g.nz + k;
    const int p = ((lx + 1) * NY + ly + 1) * NZ + lz + 1;
    const long long vx = sB[0][p], vy = sB[1][p], vz = sB[2][p];
    const long long zy = sB[2][p - NZ], zx = sB[2][p - NY * NZ], yz = sB[1][p - 1], yx = sB[1][p - NY * NZ];
    const long long xz = sB[0][p - 1], xy = sB[0][p - NZ];
    const bool layer = pm.L && (pml_row(j, g.ny, pm.L) >= 0 || pml_row(k, g.nz, pm.L) >= 0);
    int hi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) hi[c] = layer ? -1 : high_bits(pe[t][c]);
    const unsigned weak = weak_test(0, vz, zy, hi[0]) | weak_test(1, vy, yz, hi[0]) | weak_test(2, vx, xz, hi[1]) |
                          weak_test(3, vz, zx, hi[1]) | weak_test(4, vy, yx, hi[2]) | weak_test(5, vx, xy, hi[2]);
    if (j >= g.ny || k >= g.nz) continue;
    const long long yBz = scaled<2>(vz - zy, k64.fd[1]), zBy = scaled<2>(vy - yz, k64.fd[2]);
    const long long zBx = scaled<2>(vx - xz, k64.fd[2]), xBz = scaled<2>(vz - zx, k64.fd[0]);
    const long long xBy = scaled<2>(vy - yx, k64.fd[0]), yBx = scaled<2>(vx - xy, k64.fd[1]);
    const double *Hx = hb.c[0], *Hy = hb.c[1], *Hz = hb.c[2];
    if (layer) {
      CurlD<double> d;
      d.dyEz = weak & 1 ? (Hz[id] - below(Hz, g, slab, j - 1, k)) * fc.idy : fixed_to_double(yBz, sc[2]) * k64.idt;
      d.dzEy = weak & 2 ? (Hy[id] - below(Hy, g, slab, j, k - 1)) * fc.idz : fixed_to_double(zBy, sc[1]) * k64.idt;
      d.dzEx = weak & 4 ? (Hx[id] - below(Hx, g, slab, j, k - 1)) * fc.idz : fixed_to_double(zBx, sc[0]) * k64.idt;
      d.dxEz = weak & 8 ? (Hz[id] - below(Hz, g, slab_of(g, i - 1), j, k)) * fc.idx : fixed_to_double(xBz, sc[2]) * k64.idt;
      d.dxEy = weak & 16 ? (Hy[id] - below(Hy, g, slab_of(g, i - 1), j, k)) * fc.idx : fixed_to_double(xBy, sc[1]) * k64.idt;
      d.dyEx = weak & 32 ? (Hx[id] - below(Hx, g, slab, j - 1, k)) * fc.idy : fixed_to_double(yBx, sc[0]) * k64.idt;
      e_layers(g, pm, slab, j, k, d);
      f.c[EX][id] = pe[t][0] + fc.dt * ((d.dyEz - d.dzEy) - pj[t][0]);
      f.c[EY][id] = pe[t][1] + fc.dt * ((d.dzEx - d.dxEz) - pj[t][1]);
      f.c[EZ][id] = pe[t][2] + fc.dt * ((d.dxEy - d.dyEx) - pj[t][2]);
      continue;
    }
    // the difference of derivatives a and b, a - b; the one of A, B from slab s, row and
    // column down by one where it is weak
    auto put = [&](int c, long long a, int ca, const double* A, int sa, int ja, int ka, double ia, long long b, int cb,
                   const double* B, int sb, int jb, int kb, double ib) {
      const unsigned w = weak >> (2 * c) & 3u;
      double v;
      if (w) {
        const double da = w & 1 ? (A[id] - below(A, g, sa, ja, ka)) * ia : fixed_to_double(a, sc[ca]) * k64.idt;
        const double db = w & 2 ? (B[id] - below(B, g, sb, jb, kb)) * ib : fixed_to_double(b, sc[cb]) * k64.idt;
        v = pe[t][c] + fc.dt * ((da - db) - pj[t][c]);
      } else {
        const double dE = fixed_to_double(aligned_diff(a, sc[ca], b, sc[cb]), min(sc[ca], sc[cb]));
        v = pe[t][c] + fma(-fc.dt, pj[t][c], dE);
      }
      f.c[EX + c][id] = v;
    };
    const int sm = slab_of(g, i - 1);
    put(0, yBz, 2, Hz, slab, j - 1, k, fc.idy, zBy, 1, Hy, slab, j, k - 1, fc.idz);
    put(1, zBx, 0, Hx, slab, j, k - 1, fc.idz, xBz, 2, Hz, sm, j, k, fc.idx);
    put(2, xBy, 1, Hy, sm, j, k, fc.idx, yBx, 0, Hx, slab, j - 1, k, fc.idy);
  }
}

// Derivative n of curl'(E) in FP64 from global memory: the same code for every n, so
// that the lanes of a warp stay together, and the 18 loads in flight at once.
__device__ __forceinline__ double curl_term(const Geom<double>& g, const Smooth<double>& S, const Fields<double>& f,
                                            const FieldCoef<double>& fc, int n, int i, int j, int k) {
  const bool y = n == 0 || n == 5, z = n == 1 || n == 2;  // the axis of the derivative
  const double* F = n % 3 == 0 ? f.c[EZ] : (n % 3 == 1 ? f.c[EY] : f.c[EX]);
  int ox[3], oy[3], oz[3];  // offsets of the neighbours at -1, 0, 1; -1 beyond the grid
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int s = slab_of(g, i + d - 1);
    int jj = j + d - 1, kk = k + d - 1;
    if (!g.pml) {
      jj = jj < 0 ? jj + g.ny : (jj >= g.ny ? jj - g.ny : jj);
      kk = kk < 0 ? kk + g.nz : (kk >= g.nz ? kk - g.nz : kk);
    }
    ox[d] = s < 0 ? -1 : s * g.nyz;
    oy[d] = (unsigned)jj < (unsigned)g.ny ? jj * g.nz : -1;
    oz[d] = (unsigned)kk < (unsigned)g.nz ? kk : -1;
  }
  double v[2][3][3];  // along the derivative's axis, the first and the second other axis
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int oa = y ? oy[1 + p] : (z ? oz[1 + p] : ox[1 + p]), ob = y || z ? ox[q] : oy[q], oc = z ? oy[r] : oz[r];
        v[p][q][r] = (oa | ob | oc) >= 0 ? F[oa + ob + oc] : 0.0;
      }
  const double wa = y ? S.a[1] : (z ? S.a[2] : S.a[0]), w1 = y ? S.b1[1] : (z ? S.b1[2] : S.b1[0]);
  const double w2 = y ? S.b2[1] : (z ? S.b2[2] : S.b2[0]), wg = y ? S.g[1] : (z ? S.g[2] : S.g[0]);
  double m[2];
#pragma unroll
  for (int p = 0; p < 2; ++p)
    m[p] = wa * v[p][1][1] + w1 * (v[p][2][1] + v[p][0][1]) + w2 * (v[p][1][2] + v[p][1][0]) +
           wg * (v[p][2][2] + v[p][2][0] + v[p][0][2] + v[p][0][0]);
  return (m[1] - m[0]) * (y ? fc.idy : (z ? fc.idz : fc.idx));
}

// Smoothed curl and the magnetic half steps, as k_curl_tiled.
// The weak derivatives of a block are listed and then computed by as many threads,
// since a warp takes as long for one of them as for 32; the results take the place of
// the staged fields.  (A vacuum step with 4x8x32 blocks: 2.35 ms with each lane its own
// in place, 1.58 with all derivatives of a listed cell, 1.44 with the weak ones.)  A
// block with more of them than the list takes (ahead of a front, where values fall by
// decades per cell), or one that is not finite, is done in FP64 as a whole, with the
// smoothed values shared.
constexpr int kCurlCells = FB_X * FB_Y * FB_Z;
constexpr int kWeakList = 3072;  // of 6 x 1024
constexpr int kCurlFirst = 3 * FE_N > 6 * kCurlCells ? 3 * FE_N : 6 * kCurlCells;
constexpr size_t kCurl64Smem = 8 * (kCurlFirst + 2 * (size_t)(FXN + FYN + FZN));

// Index of the staged value q of a block at (bx, by, bz), or -1: beyond the grid, or
// beyond the slabs that nx cells need.
__device__ __forceinline__ int staged_index(const Geom<double>& g, int q, int bx, int by, int bz, int nx) {
  const int lz = q % FE_Z, r = q / FE_Z, ly = r % FE_Y, lx = r / FE_Y;
  int s = lx < nx + 2 ? slab_of(g, bx - 1 + lx) : -1;
  int j = by - 1 + ly, k = bz - 1 + lz;
  if (g.pml) {  // zero beyond the grid
    if (j < 0 || j >= g.ny || k < 0 || k >= g.nz) s = -1;
  } else {      // periodic; a block may exceed a small ny or nz more than once
    j = j < 0 ? j + g.ny : (j >= g.ny ? j - g.ny : j);
    k = k < 0 ? k + g.nz : (k >= g.nz ? k - g.nz : k);
    if ((unsigned)j >= (unsigned)g.ny) j = wrapi(j, g.ny);
    if ((unsigned)k >= (unsigned)g.nz) k = wrapi(k, g.nz);
  }
  return s < 0 ? -1 : s * g.nyz + j * g.nz + k;
}

// The smoothed fields of a block of nx slabs from staged values E(component, point),
// as smooth(component, point, steps along the two other axes, axis) gives them.
template <typename V, typename F>
__device__ __forceinline__ void smooth_block(V* out, int nx, F smooth) {
  constexpr int PX = FE_Y * FE_Z, PY = FE_Z;
  V *sxEy = out, *sxEz = sxEy + FXN, *syEz = sxEz + FXN, *syEx = syEz + FYN, *szEx = syEx + FYN, *szEy = szEx + FZN;
  const int tid = threadIdx.x;
  for (int q = tid; q < (nx + 1) * FB_Y * FB_Z; q += 256) {
    const int lz = q % FB_Z, r = q / FB_Z;
    const int p = (r / FB_Y + 1) * PX + (r % FB_Y + 1) * PY + lz + 1;
    sxEy[q] = smooth(1, p, PY, 1, 0);
    sxEz[q] = smooth(2, p, PY, 1, 0);
  }
  for (int q = tid; q < nx * (FB_Y + 1) * FB_Z; q += 256) {
    const int lz = q % FB_Z, r = q / FB_Z;
    const int p = (r / (FB_Y + 1) + 1) * PX + (r % (FB_Y + 1) + 1) * PY + lz + 1;
    syEz[q] = smooth(2, p, PX, 1, 1);
    syEx[q] = smooth(0, p, PX, 1, 1);
  }
  for (int q = tid; q < nx * FB_Y * (FB_Z + 1); q += 256) {
    const int lz = q % (FB_Z + 1), r = q / (FB_Z + 1);
    const int p = (r / FB_Y + 1) * PX + (r % FB_Y + 1) * PY + lz + 1;
    szEx[q] = smooth(0, p, PX, PY, 2);
    szEy[q] = smooth(1, p, PX, PY, 2);
  }
}

// A whole block of k_curl64 in FP64 arithmetic, in the same shared memory.
__device__ __forceinline__ void curl_block64(const Geom<double>& g, const Smooth<double>& S, const Fields<double>& f,
                                             const Fields<double>& hb, const FieldCoef<double>& fc, const Pml<double>& pm,
                                             int mode, int bx, int nx, int by, int bz, double* sE,
                                             const double (&pb)[kCurlCells / 256][3]) {
  const int tid = threadIdx.x;
  __syncthreads();
  for (int q = tid; q < FE_N; q += 256) {
    const int gi = staged_index(g, q, bx, by, bz, nx);
#pragma unroll
    for (int c = 0; c < 3; ++c) sE[c * FE_N + q] = gi < 0 ? 0.0 : f.c[EX + c][gi];
  }
  __syncthreads();
  double* sS = sE + kCurlFirst;
  smooth_block(sS, nx, [&](int c, int p, int a, int b, int ax) {
    const double* E = sE + c * FE_N + p;
    return S.a[ax] * E[0] + S.b1[ax] * (E[a] + E[-a]) + S.b2[ax] * (E[b] + E[-b]) +
           S.g[ax] * (E[a + b] + E[a - b] + E[-a + b] + E[-a - b]);
  });
  __syncthreads();
  const double *sxEy = sS, *sxEz = sxEy + FXN, *syEz = sxEz + FXN, *syEx = syEz + FYN, *szEx = syEx + FYN, *szEy = szEx + FZN;
#pragma unroll
  for (int t = 0; t < kCurlCells / 256; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % FB_Z, r = q / FB_Z, ly = r % FB_Y, lx = r / FB_Y;
    const int j = by + ly, k = bz + lz;
    if (lx >= nx || j >= g.ny || k >= g.nz) continue;
    const int x0 = (lx * FB_Y + ly) * FB_Z + lz, x1 = x0 + FB_Y * FB_Z;
    const int y0 = (lx * (FB_Y + 1) + ly) * FB_Z + lz, y1 = y0 + FB_Z;
    const int z0 = (lx * FB_Y + ly) * (FB_Z + 1) + lz;
    const CurlD<double> d = {(syEz[y1] - syEz[y0]) * fc.idy,     (szEy[z0 + 1] - szEy[z0]) * fc.idz,
                             (szEx[z0 + 1] - szEx[z0]) * fc.idz, (sxEz[x1] - sxEz[x0]) * fc.idx,
                             (sxEy[x1] - sxEy[x0]) * fc.idx,     (syEx[y1] - syEx[y0]) * fc.idy};
    curl_store(g, f, hb, fc, pm, mode, slab_of(g, bx + lx), j, k, d, pb[t]);
  }
}

__global__ void __launch_bounds__(256, 2)
    k_curl64(Geom<double> g, Smooth<double> S, Fields<double> f, Fields<double> hb, FieldCoef<double> fc,
             FieldConst64 k64, int mode, FieldSpan sp, Pml<double> pm) {
  if (!dyn_prologue(g)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sh[4];  // largest high words; weak derivatives
  __shared__ unsigned short list[kWeakList];
  long long* sE = reinterpret_cast<long long*>(smem_raw);  // [3][FE_X][FE_Y][FE_Z], origin (bx-1, by-1, bz-1)
  long long* sSxEy = sE + kCurlFirst;                      // [FB_X+1][FB_Y][FB_Z]
  long long* sSxEz = sSxEy + FXN;
  long long* sSyEz = sSxEz + FXN;                          // [FB_X][FB_Y+1][FB_Z]
  long long* sSyEx = sSyEz + FYN;
  long long* sSzEx = sSyEx + FYN;                          // [FB_X][FB_Y][FB_Z+1]
  long long* sSzEy = sSzEx + FZN;
  const int bx = blockIdx.z * sp.step, bx1 = min(bx + sp.width, g.nx), by = blockIdx.y * FB_Y, bz = blockIdx.x * FB_Z;
  const int tid = threadIdx.x;
  constexpr int kPer = FB_X * FB_Y * FB_Z / 256;
  int e[3];
  bool finite;
  double pb[kPer][3];  // H (mode 1) or B (mode 0) of the thread's cells
  if (tid < 4) sh[tid] = 0;
  {
    constexpr int kIt = (FE_N + 255) / 256;
    long long raw[kIt][3];
    int hmax[3] = {0, 0, 0};
#pragma unroll
    for (int t = 0; t < kIt; ++t) {
      const int gi = staged_index(g, tid + 256 * t, bx, by, bz, bx1 - bx);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        raw[t][c] = gi < 0 ? 0LL : __double_as_longlong(f.c[EX + c][gi]);
        hmax[c] = max(hmax[c], high_bits(raw[t][c]));
      }
    }
#pragma unroll
    for (int t = 0; t < kPer; ++t) {  // in flight with the staged values
      const int q = tid + 256 * t;
      const int lz = q % FB_Z, r = q / FB_Z;
      const int i = bx + r / FB_Y, j = by + r % FB_Y, k = bz + lz;
      const bool in = i < bx1 && j < g.ny && k < g.nz;
      const size_t id = in ? (size_t)slab_of(g, i) * g.nyz + (size_t)j * g.nz + k : 0;
#pragma unroll
      for (int c = 0; c < 3; ++c) pb[t][c] = mode == 1 ? hb.c[c][id] : f.c[BX + c][id];
    }
    __syncthreads();
    finite = block_scales(hmax, sh, e);
    if (finite)
#pragma unroll
      for (int t = 0; t < kIt; ++t) {
        const int q = tid + 256 * t;
        if (q < FE_N)
#pragma unroll
          for (int c = 0; c < 3; ++c) sE[c * FE_N + q] = field_fixed(raw[t][c], e[c]);
      }
  }
  if (!finite) {  // uniform over the block
    curl_block64(g, S, f, hb, fc, pm, mode, bx, bx1 - bx, by, bz, reinterpret_cast<double*>(smem_raw), pb);
    return;
  }
  __syncthreads();
  // sum over the 3x3 points around p with steps a, b, at 2^(s + 1); the products' low
  // words enter with their upper 15 bits
  smooth_block(sSxEy, bx1 - bx, [&](int c, int p, int a, int b, int ax) -> long long {
    const long long* E = sE + c * FE_N + p;
    const long long e1 = E[a] + E[-a], e2 = E[b] + E[-b];
    const long long cr = (E[a + b] + E[a - b]) + (E[-a + b] + E[-a - b]);
    const S32 x[4] = {split32(E[0]), split32(e1), split32(e2), split32(cr)};
    Acc32 s = {0LL, 1LL << 28};
    int l = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      acc32(s, x[k], k64.s[ax][k]);
      l += (x[k].lo >> 17) * k64.s17[ax][k];
    }
    s.M += (long long)l * 4;
    return (s.H << 3) + (s.M >> 29);
  });
  __syncthreads();
  double* sWeak = reinterpret_cast<double*>(smem_raw);  // [6][kCurlCells]
  unsigned weak_bits = 0;                               // six per cell of the thread
  {
    const WeakTest weak_test(e, sh, kFieldBits - 7);  // the smoothed values have twice the scale
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int q = tid + 256 * t;
      const int lz = q % FB_Z, r = q / FB_Z, ly = r % FB_Y, lx = r / FB_Y;
      const int i = bx + lx, j = by + ly, k = bz + lz;
      if (i >= bx1) continue;  // uniform over a warp
      const int x0 = (lx * FB_Y + ly) * FB_Z + lz, x1 = x0 + FB_Y * FB_Z;
      const int y0 = (lx * (FB_Y + 1) + ly) * FB_Z + lz, y1 = y0 + FB_Z;
      const int z0 = (lx * FB_Y + ly) * (FB_Z + 1) + lz;
      const bool layer = pm.L && (pml_row(j, g.ny, pm.L) >= 0 || pml_row(k, g.nz, pm.L) >= 0);
      int hi[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) hi[c] = layer ? -1 : high_bits(pb[t][c]);
      const unsigned weak = weak_test(0, sSyEz[y1], sSyEz[y0], hi[0]) | weak_test(1, sSzEy[z0 + 1], sSzEy[z0], hi[0]) |
                      weak_test(2, sSzEx[z0 + 1], sSzEx[z0], hi[1]) | weak_test(3, sSxEz[x1], sSxEz[x0], hi[1]) |
                      weak_test(4, sSxEy[x1], sSxEy[x0], hi[2]) | weak_test(5, sSyEx[y1], sSyEx[y0], hi[2]);
      if (j < g.ny && k < g.nz) weak_bits |= weak << (6 * t);
    }
    if (weak_bits) {
      int pos = atomicAdd(sh + 3, __popc(weak_bits));
      for (unsigned m = weak_bits; m; m &= m - 1, ++pos) {
        const int t = (__ffs(m) - 1) / 6, n = (__ffs(m) - 1) % 6, q = tid + 256 * t;
        if (pos < kWeakList) list[pos] = (unsigned short)(n * kCurlCells + q);
      }
    }
    static_assert(6 * kPer <= 32, "six bits per cell");
    static_assert(6 * kCurlCells <= 65536, "16-bit entries");
    __syncthreads();
    const int nweak = sh[3];  // uniform over the block
    if (nweak > kWeakList) {
      curl_block64(g, S, f, hb, fc, pm, mode, bx, bx1 - bx, by, bz, reinterpret_cast<double*>(smem_raw), pb);
      return;
    }
    if (nweak > 0) {
#pragma unroll 1
      for (int m = tid; m < nweak; m += 256) {
        const int n = list[m] / kCurlCells, q = list[m] % kCurlCells, r = q / FB_Z;
        sWeak[n * kCurlCells + q] = curl_term(g, S, f, fc, n, bx + r / FB_Y, by + r % FB_Y, bz + q % FB_Z);
      }
      __syncthreads();
    }
  }
  int sc[3];  // scale of the products
#pragma unroll
  for (int c = 0; c < 3; ++c) sc[c] = kFieldBits + 1023 - e[c];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int q = tid + 256 * t;
    const int lz = q % FB_Z, r = q / FB_Z, ly = r % FB_Y, lx = r / FB_Y;
    const int i = bx + lx, j = by + ly, k = bz + lz;
    if (i >= bx1 || j >= g.ny || k >= g.nz) continue;
    const int x0 = (lx * FB_Y + ly) * FB_Z + lz, x1 = x0 + FB_Y * FB_Z;
    const int y0 = (lx * (FB_Y + 1) + ly) * FB_Z + lz, y1 = y0 + FB_Z;
    const int z0 = (lx * FB_Y + ly) * (FB_Z + 1) + lz;
    const int slab = slab_of(g, i);
    const size_t id = (size_t)slab * g.nyz + (size_t)j * g.nz + k;
    // dt/2 times D_y S_y Ez, D_z S_z Ey; D_z S_z Ex, D_x S_x Ez; D_x S_x Ey, D_y S_y Ex
    const long long yEz = scaled<1>(sSyEz[y1] - sSyEz[y0], k64.hd[1]), zEy = scaled<1>(sSzEy[z0 + 1] - sSzEy[z0], k64.hd[2]);
    const long long zEx = scaled<1>(sSzEx[z0 + 1] - sSzEx[z0], k64.hd[2]), xEz = scaled<1>(sSxEz[x1] - sSxEz[x0], k64.hd[0]);
    const long long xEy = scaled<1>(sSxEy[x1] - sSxEy[x0], k64.hd[0]), yEx = scaled<1>(sSyEx[y1] - sSyEx[y0], k64.hd[1]);
    double dB[3];
    const int jr = pm.L ? pml_row(j, g.ny, pm.L) : -1, kr = pm.L ? pml_row(k, g.nz, pm.L) : -1;
    const unsigned weak = (weak_bits >> (6 * t)) & 63u;
    if (weak || jr >= 0 || kr >= 0) {  // the derivatives as doubles
      CurlD<double> d;
      d.dyEz = fixed_to_double(yEz, sc[2]) * k64.ihdt;
      d.dzEy = fixed_to_double(zEy, sc[1]) * k64.ihdt;
      d.dzEx = fixed_to_double(zEx, sc[0]) * k64.ihdt;
      d.dxEz = fixed_to_double(xEz, sc[2]) * k64.ihdt;
      d.dxEy = fixed_to_double(xEy, sc[1]) * k64.ihdt;
      d.dyEx = fixed_to_double(yEx, sc[0]) * k64.ihdt;
      if (weak & 1) d.dyEz = sWeak[q];
      if (weak & 2) d.dzEy = sWeak[kCurlCells + q];
      if (weak & 4) d.dzEx = sWeak[2 * kCurlCells + q];
      if (weak & 8) d.dxEz = sWeak[3 * kCurlCells + q];
      if (weak & 16) d.dxEy = sWeak[4 * kCurlCells + q];
      if (weak & 32) d.dyEx = sWeak[5 * kCurlCells + q];
      if (jr >= 0 || kr >= 0) curl_layers(g, pm, mode, slab, j, k, d);  // y and z at half nodes
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
