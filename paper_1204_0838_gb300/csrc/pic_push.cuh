// pic_push.cuh -- what the FP32 and FP64 particle pushes share: the layout of
// a tile's fields and current in shared memory, and the ranking of a tile's
// particles per cell.  One CTA takes one tile, its particles in passes of up to
// kChunk:
//   stage E, B; in passes: rank the particles per cell and list them in (rank,
//   cell) order; gather, push, move, writing the moved particles in that order to
//   the second buffer; then turn the staged fields' memory into the J tile; in
//   passes: deposit the particles that stayed in their cell, then the others; add
//   the tile to J, once, whatever the number of passes: each add rounds.
// A tile of more than one pass keeps the passes' lists in global memory between
// the two phases, in the cells and momenta of the first buffer, which nothing
// reads any more in the step.
// In (rank, cell) order the lanes of a warp hold distinct neighbouring cells,
// so that their reads and adds at one offset from their own cells collide
// little, and the writes are coalesced and nearly sorted for the next step.
#pragma once

#include "pic_tiled.cuh"

namespace pic {

constexpr int kPushThreads = 256;  // per SM: FP32 three CTAs at 80 registers, FP64 two at 128
constexpr int kChunk = 2304;       // particles per pass over a tile (FP32: the lists that fit three CTAs)
constexpr int kRanks = 32;         // ranks per cell that are ordered; later ones follow in any order
// entry of the order list: particle of the pass (12 bits), cell slot (12
// bits), cell steps + 1 per axis (6 bits) and two flags
constexpr unsigned kCross = 1u << 31;  // not with the ordered particles: alone (listed) or not at all
constexpr unsigned kStray = 1u << 30;  // outside the tile: dropped, error bit set
constexpr unsigned kSteps = 63u << 24;  // the cell steps; all set (no particle's steps): push again

// The shared-memory region.  Components are stored with their axes rotated,
// [i_d][i_e][i_f] with (e, f) the axes after d in cyclic order, so that one
// body serves the three rotations with the same offsets (three unrolled bodies
// overflow the instruction cache): two field components per d, in T or 64-bit
// words, and J as [d][words of a sum] in 32-bit words (FP32 2, FP64 3).  FIXED:
// tiles of up to 8 cells per axis, strides known to the compiler; otherwise any tile, with
// odd pitches of rows and planes (a warp's cells along z lie a plane apart in one of the
// rotations, and an even pitch put them on few banks: two FP32 steps of 14 M
// particles on 4x8x16 tiles 10.5 -> 5.9 ms, on 16x8x8 7.8 -> 6.8; on 8x8x8 fixed 5.0).  The fixed
// strides are the best of a search over shapes of a warp's 32 cells and pitches:
// 1x8x4 cells (slot order) read 32-bit fields and add to J in 1, 2 and 1 (fields)
// or 2, 1 and 1 (J) wavefronts for the three rotations, and read 64-bit fields,
// where each lane starts at its own half cell, in 1.72 per half warp (linear
// cell order with one pitch: 5/3 and 2.13).
template <typename T, bool FIXED>
struct PushLayout {
  int t[3];
  __host__ __device__ explicit PushLayout(const Tiles& tl) : t{tl.tx, tl.ty, tl.tz} {}
  // pad = 4: staged fields, 5: J
  __host__ __device__ __forceinline__ int se(int d, int pad) const { return FIXED ? 8 + pad : (t[(d + 2) % 3] + pad) | 1; }
  __host__ __device__ __forceinline__ int sd(int d, int pad) const {
    if (!FIXED) return (t[(d + 1) % 3] + pad) * se(d, pad) | 1;
    if (pad == 5) return d == 0 ? 169 : (d == 1 ? 172 : 184);
    return d == 0 ? 144 : (sizeof(T) == 8 ? (d == 1 ? 149 : 148) : (d == 1 ? 145 : 152));
  }
  __host__ __device__ __forceinline__ int part(int d, int pad) const {
    return FIXED ? (8 + pad) * sd(d, pad) : (t[d] + pad) * sd(d, pad);
  }
  static constexpr int kJWords = sizeof(T) == 8 ? 3 : 2;
  __host__ __device__ __forceinline__ int start(int d, int pad) const {
    const int n = pad == 4 ? 2 : kJWords;
    return d == 0 ? 0 : n * (part(0, pad) + (d == 1 ? 0 : part(1, pad)));
  }
  __host__ __device__ int region(int pad) const {
    return (pad == 4 ? 2 : kJWords) * (part(0, pad) + part(1, pad) + part(2, pad));
  }
  // cell slots: a warp's 32 are 1x8x4 cells (fixed) or consecutive cells
  __host__ __device__ int words() const { return FIXED ? 2 * t[0] : (t[0] * t[1] * t[2] + 31) / 32; }
  __device__ __forceinline__ int slot(int lx, int ly, int lz) const {
    return FIXED ? (lx * 2 + (lz >> 2)) * 32 + ly * 4 + (lz & 3) : (lx * t[1] + ly) * t[2] + lz;
  }
  __device__ __forceinline__ void cell(int s, int (&l)[3]) const {
    if (FIXED) {
      l[0] = s >> 6;
      l[1] = (s >> 2) & 7;
      l[2] = ((s >> 3) & 4) | (s & 3);
    } else {
      l[0] = s / (t[1] * t[2]);
      const int r = s - l[0] * t[1] * t[2];
      l[1] = r / t[2];
      l[2] = r - l[1] * t[2];
    }
  }
};

// Shared memory: the region (staged fields and the ranking's scratch, then J),
// the order list (32-bit entries), the FP32 pair list, the list of particles
// that deposit alone, the wrapped grid offsets per axis, and 64 ints of scalars.
struct PushSmem {
  size_t hist, mask, base, order, pair, cross, tab, scal, total;
  template <typename T, bool FIXED>
  __host__ __device__ static PushSmem of(const Tiles& tl) {
    const PushLayout<T, FIXED> L(tl);
    PushSmem s;
    const size_t w = L.words();
    size_t a = ((size_t)L.region(4) * sizeof(T) + 15) / 16 * 16;
    s.hist = a;
    a += 4 * 32 * w;
    s.mask = a;
    a += 4 * kRanks * w;
    s.base = a;
    a += (2 * kRanks * w + 15) / 16 * 16;
    const size_t j = (size_t)L.region(5) * 4;
    a = ((a > j ? a : j) + 15) / 16 * 16;
    s.order = a;
    a += 4 * (size_t)kChunk;
    s.pair = a;
    if (sizeof(T) == 4) a += 2 * (size_t)kChunk;  // FP64 takes the particles one by one
    s.cross = a;
    a += 2 * (size_t)kChunk;
    s.tab = a;
    a += 4 * (size_t)(tl.tx + tl.ty + tl.tz + 15);
    s.scal = (a + 15) / 16 * 16;
    s.total = s.scal + 4 * 64;
    return s;
  }
};

// Pointers into the shared memory of a CTA, and the scalars: [0] particles
// without an ordered rank, [1] particles that deposit alone, [2, 4) sums or
// maxima over the tile, [4, 7) J scale per component, [7] whether particles of the
// pass are to be pushed again on their own (FP32), [8, 16) scan partials,
// [16, 33) first pair of each pair of ranks, [33] ordered particles, [34, 50)
// first position of each pair of ranks, [50, 62) field scales (FP64), [50, 53)
// scale of P per component and [53] the weight below which a particle is light (FP32).
// All but [2, 8) and [50, 64) belong to a pass.
constexpr int kPassScalars = 50;
struct PushTile {
  int* hist;
  unsigned* mask;         // [rank][word]: cells that hold more than `rank` particles
  unsigned short* base;   // [rank][word]: position of the word's first particle
  unsigned* order;
  unsigned short* cross;
  int *tabx, *taby, *tabz;  // wrapped grid offsets of the staged cells
  int* sc;
  int x0, y0, z0;         // tile corner (cells)

  // position of rank r of the cell in slot s
  __device__ __forceinline__ int position(int W, int r, int s) const {
    const int i = r * W + (s >> 5);
    return base[i] + __popc(mask[i] & ((1u << (s & 31)) - 1u));
  }
};

template <typename T, bool FIXED>
__device__ __forceinline__ PushTile push_tile(unsigned char* smem, const Geom<T>& g, const Tiles& tl, int t) {
  const PushSmem so = PushSmem::of<T, FIXED>(tl);
  PushTile P;
  P.hist = reinterpret_cast<int*>(smem + so.hist);
  P.mask = reinterpret_cast<unsigned*>(smem + so.mask);
  P.base = reinterpret_cast<unsigned short*>(smem + so.base);
  P.order = reinterpret_cast<unsigned*>(smem + so.order);
  P.cross = reinterpret_cast<unsigned short*>(smem + so.cross);
  P.tabx = reinterpret_cast<int*>(smem + so.tab);
  P.taby = P.tabx + tl.tx + 5;
  P.tabz = P.taby + tl.ty + 5;
  P.sc = reinterpret_cast<int*>(smem + so.scal);
  const int rest = t / tl.ntz;
  if (threadIdx.x < 64) P.sc[threadIdx.x] = 0;
  P.x0 = (rest / tl.nty) * tl.tx;
  P.y0 = (rest % tl.nty) * tl.ty;
  P.z0 = (t % tl.ntz) * tl.tz;
  // origin tile - 2; J reaches one cell further than E, B
  for (int i = threadIdx.x; i < tl.tx + tl.ty + tl.tz + 15; i += kPushThreads) {
    int v;
    if (i < tl.tx + 5)
      v = wrapi(P.x0 - 2 + i, g.nx) * g.nyz;
    else if (i < tl.tx + tl.ty + 10)
      v = wrapi(P.y0 - 2 + i - (tl.tx + 5), g.ny) * g.nz;
    else
      v = wrapi(P.z0 - 2 + i - (tl.tx + tl.ty + 10), g.nz);
    P.tabx[i] = v;
  }
  return P;
}

// Clear the ranking's scratch for a pass (a barrier must follow; the tile's
// scalars are cleared once).
__device__ __forceinline__ void rank_clear(const PushTile& P, int W) {
  for (int i = threadIdx.x; i < 32 * W; i += kPushThreads) P.hist[i] = 0;
  for (int i = threadIdx.x; i < kRanks * W; i += kPushThreads) P.mask[i] = 0u;
  if (threadIdx.x < 3) P.sc[threadIdx.x < 2 ? threadIdx.x : 7] = 0;
}

// Particles [begin, begin + n) of pass ps of npass over a tile of ntile: sizes
// within one of each other, so that none of several passes is below kChunk / 2.
struct Pass {
  int begin, n;
  __device__ __forceinline__ Pass(int ps, int npass, int ntile) {
    const int per = ntile / npass, more = ntile - per * npass;
    begin = ps * per + min(ps, more);
    n = per + (ps < more ? 1 : 0);
  }
};

// Keep a pass's lists: the order list in its cells, the pairs (nitem entries, or
// none), the particles that deposit alone and the scalars in its momenta.  Barriers
// before and after.
template <typename T>
__device__ __forceinline__ void keep_lists(const PushTile& P, const Parts<T>& p, int c0, int nch, int nitem,
                                           const unsigned short* pair) {
  unsigned *c = reinterpret_cast<unsigned*>(p.cell + c0), *u0 = reinterpret_cast<unsigned*>(p.u[0] + c0),
           *u1 = reinterpret_cast<unsigned*>(p.u[1] + c0), *u2 = reinterpret_cast<unsigned*>(p.u[2] + c0);
  for (int i = threadIdx.x; i < nch; i += kPushThreads) c[i] = P.order[i];
  for (int i = threadIdx.x; i < nitem; i += kPushThreads) u0[i] = pair[i];
  for (int i = threadIdx.x; i < P.sc[1]; i += kPushThreads) u1[i] = P.cross[i];
  if (threadIdx.x < kPassScalars) u2[threadIdx.x] = (unsigned)P.sc[threadIdx.x];
}
// Bring them back (from L2: the cells were read through other paths before).
template <typename T>
__device__ __forceinline__ void fetch_lists(const PushTile& P, const Parts<T>& p, int c0, int nch,
                                            unsigned short* pair) {
  const unsigned *c = reinterpret_cast<unsigned*>(p.cell + c0), *u0 = reinterpret_cast<unsigned*>(p.u[0] + c0),
                 *u1 = reinterpret_cast<unsigned*>(p.u[1] + c0), *u2 = reinterpret_cast<unsigned*>(p.u[2] + c0);
  const int n1 = (int)__ldcg(u2 + 1);
  for (int i = threadIdx.x; i < nch; i += kPushThreads) {
    P.order[i] = __ldcg(c + i);
    if (pair) pair[i] = (unsigned short)__ldcg(u0 + i);
    if (i < n1) P.cross[i] = (unsigned short)__ldcg(u1 + i);
  }
  if (threadIdx.x < kPassScalars && !(threadIdx.x >= 2 && threadIdx.x < 8)) P.sc[threadIdx.x] = (int)__ldcg(u2 + threadIdx.x);
}

constexpr int kPerThread = kChunk / kPushThreads;

// Constants of a push that cost divisions, formed on the host.
template <typename T>
struct PushCoef {
  T h;       // q dt / (2 m)
  T q;
  T dtd[3];  // dt / d
  T jc[3];   // -1 / (dt d_e d_f)
};

__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// The (x, y) rows of a halo of ny rows per slab that a half warp takes, 16 rows
// apart: no division per row.
struct RowWalk {
  int lx, ly, ny, qx, qy;
  __device__ __forceinline__ explicit RowWalk(int n) : ny(n), qx(16 / n), qy(16 % n) {
    const int r = threadIdx.x >> 4;
    lx = r / n;
    ly = r % n;
  }
  __device__ __forceinline__ void next() {
    lx += qx;
    ly += qy;
    if (ly >= ny) {
      ly -= ny;
      lx += 1;
    }
  }
};
static_assert(kPushThreads == 256, "RowWalk: 16 half warps");

// Count the pass's particles [c0, c0 + nch) per cell: sr[] = slot and rank of
// this thread's particles (-2: outside the tile).  A barrier must follow.
template <typename T, bool FIXED>
__device__ __forceinline__ void rank_count(const PushTile& P, const PushLayout<T, FIXED>& L, const Geom<T>& g,
                                           const Tiles& tl, const int* __restrict__ cells, int c0, int nch,
                                           int (&sr)[kPerThread], int* err) {
  const float inv_nyz = 1.0f / (float)g.nyz, inv_nz = 1.0f / (float)g.nz;
#pragma unroll
  for (int it = 0; it < kPerThread; ++it) {
    const int k = it * kPushThreads + threadIdx.x;
    sr[it] = -1;
    if (k < nch) {
      // cell - (tile corner) split by quotient estimates, then checked exactly
      const int rel = cells[c0 + k] - P.x0 * g.nyz - P.y0 * g.nz - P.z0;
      int lx = __float2int_rn((float)rel * inv_nyz);
      int rem = rel - lx * g.nyz;
      if (rem < 0) {
        lx -= 1;
        rem += g.nyz;
      }
      int ly = __float2int_rn((float)rem * inv_nz);
      int lz = rem - ly * g.nz;
      if (lz < 0) {
        ly -= 1;
        lz += g.nz;
      }
      const bool in = lx >= 0 && lx < tl.tx && ly >= 0 && ly < tl.ty && lz >= 0 && lz < tl.tz &&
                      (lx * g.ny + ly) * g.nz + lz == rel;
      if (in) {
        const int s = L.slot(lx, ly, lz);
        sr[it] = s | (atomicAdd(P.hist + s, 1) << 12);
      } else {  // never expected: keeps every index in range
        atomicOr(err, 4);
        sr[it] = -2;
      }
    }
  }
}

// Occupancy of every rank: bit of a slot set in mask[r][word] if the cell holds
// more than r particles.  A barrier must follow.
__device__ __forceinline__ void rank_masks(const PushTile& P, int W) {
  for (int i = threadIdx.x; i < 32 * W; i += kPushThreads) {
    const int n = min(P.hist[i], kRanks);
    for (int r = 0;; ++r) {
      const unsigned m = __ballot_sync(0xffffffffu, n > r);
      if (!m) break;
      if ((threadIdx.x & 31) == 0) P.mask[r * W + (i >> 5)] = m;
    }
  }
}

// Positions: an exclusive scan of the populations over (rank, word), then the
// order list.  Ends with the list written (a barrier must follow).
__device__ __forceinline__ void rank_order(const PushTile& P, int W, int nch, const int (&sr)[kPerThread]) {
  const int tid = threadIdx.x, lane = tid & 31;
  {
    const int n = kRanks * W, per = (n + kPushThreads - 1) / kPushThreads;
    const int b = min(tid * per, n), e = min(b + per, n);
    int s = 0;
    for (int i = b; i < e; ++i) s += __popc(P.mask[i]);
    int incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) P.sc[8 + (tid >> 5)] = incl;
    __syncthreads();
    int run = incl - s;
    for (int k = 0; k < (tid >> 5); ++k) run += P.sc[8 + k];
    for (int i = b; i < e; ++i) {
      P.base[i] = (unsigned short)run;
      run += __popc(P.mask[i]);
    }
    if (tid == kPushThreads - 1) P.sc[33] = run;
  }
  __syncthreads();
  const int ranked = P.sc[33];
#pragma unroll
  for (int it = 0; it < kPerThread; ++it) {
    const int k = it * kPushThreads + tid;
    if (k < nch) {
      const int v = sr[it], s = v & 4095, r = v >> 12;
      const bool stray = v == -2;
      const int pos = !stray && r < kRanks ? P.position(W, r, s) : ranked + atomicAdd(P.sc, 1);
      P.order[pos] = stray ? (unsigned)k | kStray : (unsigned)k | ((unsigned)s << 12);
    }
  }
}

// Store a moved particle's cell and key.  l: its cell in the tile, dc: its
// steps (at most one cell per axis, periodic in the storage frame).  Returns
// the destination tile or -1 (absorbed), and lists a particle that left its
// cell, or that deposits alone for another reason, at position pos.
template <typename T>
__device__ __forceinline__ int place_moved(const PushTile& P, const Geom<T>& g, const Tiles& tl, int t,
                                           const int (&l)[3], const int (&dc)[3], bool good, bool alone, int origin_after,
                                           int xlo, int xhi, int pos, unsigned ent, int* cell_out, int* key_out) {
  int n0 = P.x0 + l[0] + dc[0], n1 = P.y0 + l[1] + dc[1], n2 = P.z0 + l[2] + dc[2];
  int key = t;
  if ((dc[0] | dc[1] | dc[2]) || alone) {
    n0 = wrapi(n0, g.nx), n1 = wrapi(n1, g.ny), n2 = wrapi(n2, g.nz);
    if ((unsigned)(n0 - P.x0) >= (unsigned)tl.tx || (unsigned)(n1 - P.y0) >= (unsigned)tl.ty ||
        (unsigned)(n2 - P.z0) >= (unsigned)tl.tz)
      key = tile_of(g, tl, n0, n1, n2);
    P.order[pos] = ent | kCross | ((unsigned)(dc[0] + 1) << 24) | ((unsigned)(dc[1] + 1) << 26) |
                   ((unsigned)(dc[2] + 1) << 28);
    P.cross[atomicAdd(P.sc + 1, 1)] = (unsigned short)pos;
  }
  *cell_out = (n0 * g.ny + n1) * g.nz + n2;
  if (!g.periodic_x) {
    int rel = n0 - origin_after;
    if (rel < 0) rel += g.nx;
    if (rel < xlo || rel > xhi) key = -1;
  }
  // absorbing layers: a particle that leaves the y, z cells [L, n - L) is absorbed
  if (g.pml && (n1 < g.pml || n1 >= g.ny - g.pml || n2 < g.pml || n2 >= g.nz - g.pml)) key = -1;
  if (!good) {  // absorbed without moving or depositing
    key = -1;
    P.order[pos] = ent | kCross;
  }
  *key_out = key;
  return key;
}

// Count the particles that leave for other tiles (all 32 lanes call).
__device__ __forceinline__ void count_leaving(int* cnt_next, int key, int t) {
  const int k = key == t ? -2 : key;
  if (__any_sync(0xffffffffu, k >= 0)) warp_count(cnt_next, k, false, nullptr);
}

}  // namespace pic
