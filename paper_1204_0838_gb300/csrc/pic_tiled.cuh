// pic_tiled.cuh -- particles are kept grouped by cell tile: tile geometry, and
// the re-binning after each step, a counting sort by tile (counts from the
// push, scan, scatter).  The push itself is in pic_push32.cuh and pic_push64.cuh.
#pragma once

#include "pic_fixed64.cuh"
#include "pic_kernels.cuh"

namespace pic {

template <typename T>
__device__ __forceinline__ int tile_of(const Geom<T>& g, const Tiles& tl, int cx, int cy, int cz) {
  return ((cx / tl.tx) * tl.nty + cy / tl.ty) * tl.ntz + cz / tl.tz;
}

// Shared-memory extents: E/B staged over cells [c0-2, c0+t+2) per axis (the
// half-staggered cubic gather reaches c-2 .. c+2), J over [c0-2, c0+t+3)
// (the Esirkepov window of a particle that moves at most one cell reaches
// c-2 .. c+3).
__host__ __device__ __forceinline__ int stage_n(const Tiles& tl) { return (tl.tx + 4) * (tl.ty + 4) * (tl.tz + 4); }
__host__ __device__ __forceinline__ int jtile_n(const Tiles& tl) { return (tl.tx + 5) * (tl.ty + 5) * (tl.tz + 5); }

// The size that a handle accepts tiles by (at most 227 KB): the staged fields,
// the J tile and FP32's ordering scratch side by side.  The push itself needs
// less, since its J tile takes the place of the staged fields.
template <typename T>
size_t tiled_smem_bytes(const Tiles& tl) {
  const size_t b = sizeof(T) * 6 * (size_t)stage_n(tl) + 8 * 3 * (size_t)jtile_n(tl);
  return sizeof(T) == 4 ? b + 4 * ((size_t)tl.tx * tl.ty * tl.tz + 100) + 4096 : b + 72;
}

__device__ __forceinline__ void red_u32(unsigned* a, unsigned v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(a)), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Warp-aggregated add of 1 to counter[key] for every lane with key >= 0;
// returns this lane's rank among the lanes that share its key, and the
// aggregated base offset through *base (only meaningful if want_base).
// All 32 lanes must call it.
__device__ __forceinline__ int warp_count(int* counter, int key, bool want_base, int* base) {
  const unsigned m = __match_any_sync(0xffffffffu, key);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  int b = 0;
  if (lane == leader && key >= 0) b = want_base ? atomicAdd(counter + key, __popc(m)) : (atomicAdd(counter + key, __popc(m)), 0);
  b = __shfl_sync(0xffffffffu, b, leader);
  if (base) *base = b;
  return __popc(m & lanemask_lt());
}

// Comparisons of an offset against 0 and 1, on the bit pattern with integer
// instructions, off the slow FP64 pipe: for doubles of either sign the int64
// view orders non-negative values like the values and makes every negative
// value (and -0) negative.
__device__ __forceinline__ bool lt_zero(double o) { return __double_as_longlong(o) < 0; }
__device__ __forceinline__ bool ge_one(double o) { return __double_as_longlong(o) >= 0x3FF0000000000000LL; }

// Keys from the current cells (used after loading or set_particles).
template <typename T>
__global__ void k_keys(Geom<T> g, Tiles tl, Parts<T> p, const int* __restrict__ d_np, int* keys, int* cnt) {
  const int n = *d_np;
  for (int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
    const int pi = base + threadIdx.x;
    int key = -2;
    if (pi < n) {
      const int cell = p.cell[pi];
      const int cx = cell / g.nyz, r = cell - cx * g.nyz;
      key = tile_of(g, tl, cx, r / g.nz, r - (r / g.nz) * g.nz);
      keys[pi] = key;
    }
    warp_count(cnt, key, false, nullptr);
  }
}

// Exclusive scan of the tile counts into tile starts, 4096 tiles per CTA, four
// per thread.  With more than one CTA, k_tile_sums gives the CTAs' sums first,
// and each CTA adds up those before it.  Starts are clamped to the capacity; a
// total above it sets the capacity error bit.  (One CTA with a strided chunk per
// thread took 380 us for 196,608 tiles; the two kernels take 8.)
constexpr int kScanTiles = 4096;

__device__ __forceinline__ long long block_sum_ll(long long v, long long* part) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  v = part[threadIdx.x & 31];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  return v;
}

static __global__ void __launch_bounds__(1024) k_tile_sums(const int* __restrict__ cnt, int n,
                                                           long long* __restrict__ sums) {
  __shared__ long long part[32];
  long long v = 0;
  for (int k = 0; k < kScanTiles / 1024; ++k) {
    const int i = blockIdx.x * kScanTiles + k * 1024 + threadIdx.x;
    if (i < n) v += cnt[i];
  }
  v = block_sum_ll(v, part);
  if (threadIdx.x == 0) sums[blockIdx.x] = v;
}

static __global__ void __launch_bounds__(1024) k_scan_tiles(const int* __restrict__ cnt, int* __restrict__ tstart,
                                                            int n, const long long* __restrict__ sums, int* d_np_out,
                                                            int capacity, int* err) {
  __shared__ long long part[32];
  const int tid = threadIdx.x, lane = tid & 31;
  long long before = 0;
  for (int b = tid; b < (int)blockIdx.x; b += 1024) before += sums[b];
  if (blockIdx.x > 0) before = block_sum_ll(before, part);
  const int i0 = blockIdx.x * kScanTiles + 4 * tid;
  int c[4];
  long long s = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    c[k] = i0 + k < n ? cnt[i0 + k] : 0;
    s += c[k];
  }
  long long incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) part[tid >> 5] = incl;
  __syncthreads();
  long long run = before + incl - s;
  for (int k = 0; k < (tid >> 5); ++k) run += part[k];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i0 + k < n) tstart[i0 + k] = (int)min(run, (long long)capacity);
    run += c[k];
    if (i0 + k == n - 1) {
      tstart[n] = (int)min(run, (long long)capacity);
      *d_np_out = (int)min(run, (long long)capacity);
      if (run > capacity) atomicOr(err, 1);
    }
  }
}

// Scatter the kept particles into their tiles of the other buffer.
template <typename T>
__global__ void k_scatter(Parts<T> src, const int* __restrict__ keys, const int* __restrict__ d_np_src, int capacity,
                          Parts<T> dst, const int* __restrict__ tstart, int* fill, int* err) {
  const int n = min(*d_np_src, capacity);
  for (int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
    const int pi = base + threadIdx.x;
    const int key = pi < n ? keys[pi] : -2;
    // read the record before reserving its slot, so that these loads overlap
    // the reservation's atomic round trip instead of following it
    int cell = 0;
    T o[3] = {T(0), T(0), T(0)}, u[3] = {T(0), T(0), T(0)}, w = T(0);
    uint32_t id = 0;
    if (key >= 0) {
      cell = src.cell[pi];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        o[d] = src.o[d][pi];
        u[d] = src.u[d][pi];
      }
      w = src.w[pi];
      if (src.id) id = src.id[pi];
    }
    int off;
    const int rank = warp_count(fill, key, true, &off);
    if (key >= 0) {
      const int slot = tstart[key] + off + rank;
      if (slot >= tstart[key + 1]) {
        atomicOr(err, 2);
        continue;
      }
      dst.cell[slot] = cell;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        dst.o[d][slot] = o[d];
        dst.u[d][slot] = u[d];
      }
      dst.w[slot] = w;
      if (dst.id) dst.id[slot] = id;
    }
  }
}

// Window injection into a tile-sorted buffer: pass 0 counts per tile into
// cnt, pass 1 places the particles with the tile fill counters.  The draws
// are the same counter-based SplitMix64 keys as plain loading, so both
// passes regenerate identical particles.
template <typename T>
__global__ void k_inject_tiled(Geom<T> g, Tiles tl, Parts<T> p, LoadSpec L, int pass, int* cnt,
                               const int* __restrict__ tstart, int* fill, int* err) {
  if (!dyn_prologue(g)) return;
  if (g.dyn) L.shifts = g.dyn->shifts;
  const long long nslot = (long long)(L.hi - L.lo + 1) * g.nyz * L.ppc;
  for (long long q0 = (long long)blockIdx.x * blockDim.x; q0 < nslot; q0 += (long long)gridDim.x * blockDim.x) {
    const long long qq = q0 + threadIdx.x;
    int key = -2;
    double o[3] = {0, 0, 0}, n = 0;
    int sx = 0, j = 0, k = 0, sl = 0;
    unsigned long long cell = 0;
    if (qq < nslot) {
      sl = (int)(qq % L.ppc);
      const long long c = qq / L.ppc;
      const int r = (int)(c % g.nyz);
      const int ci = L.lo + (int)(c / g.nyz);
      j = r / g.nz;
      k = r - j * g.nz;
      const long long lab = L.shifts + ci;
      cell = ((unsigned long long)lab * g.ny + j) * g.nz + k;
      const unsigned long long ctr = (cell * L.ppc + sl) * 3ull;
      double rr[3];
      for (int d = 0; d < 3; ++d) rr[d] = unit_uniform(L.seed, ctr + d);
      if (L.lattice) {
        const int ix = sl / (L.ns[1] * L.ns[2]), iy = (sl / L.ns[2]) % L.ns[1], iz = sl % L.ns[2];
        o[0] = (ix + rr[0]) / L.ns[0];
        o[1] = (iy + rr[1]) / L.ns[1];
        o[2] = (iz + rr[2]) / L.ns[2];
      } else {
        o[0] = rr[0];
        o[1] = rr[1];
        o[2] = rr[2];
      }
      const bool inner = j >= L.pml && j < g.ny - L.pml && k >= L.pml && k < g.nz - L.pml;
      n = inner ? profile_at(L.px, L.pn, L.np, L.x0 + ((double)lab + o[0]) * L.dx) : 0.0;
      sx = slab_of(g, ci);
      if (n > 0.0) key = tile_of(g, tl, sx, j, k);
    }
    if (pass == 0) {
      warp_count(cnt, key, false, nullptr);
      continue;
    }
    int off;
    const int rank = warp_count(fill, key, true, &off);
    if (key >= 0) {
      const int slot = tstart[key] + off + rank;
      if (slot >= tstart[key + 1]) {
        atomicOr(err, 2);
        continue;
      }
      p.cell[slot] = sx * g.nyz + j * g.nz + k;
      for (int d = 0; d < 3; ++d) {
        T od = (T)o[d];
        if (od >= T(1)) od = one_below<T>();
        p.o[d][slot] = od;
        p.u[d][slot] = T(0);
      }
      p.w[slot] = (T)(n * L.dVppc);
      if (p.id) p.id[slot] = (uint32_t)(cell * L.ppc + sl);
    }
  }
}

}  // namespace pic
