// pic_push32.cuh -- the FP32 particle push: gather, Boris push, move and
// Esirkepov deposit of one cell tile per CTA.
//
// What bounded the one-pass kernel that this replaces: shared-memory
// wavefronts (L1tex 75-80 % busy, two thirds of them bank conflicts), because
// every particle read its own 4x4x4 windows at a start that depends on the
// half cell it sits in, and added 2 x 144 words of its own to the J tile.
// What this kernel does about it:
// - Two particles of one cell per thread.  The particles of a tile are ranked
//   per cell; a thread takes ranks 2k and 2k + 1 of a cell.  The two share
//   every field load of the gather (the union window: 5 nodes along
//   half-staggered axes with a zero weight at one end, 540 loads per pair
//   instead of 768) and every add of the deposit (one exact integer sum per
//   node and pair).
// - Every lane reads and adds at the same offset from its own cell, so that
//   bank conflicts depend on the cells alone; the lanes of a warp hold
//   neighbouring cells.
// - Two phases over one shared-memory region: all particles gather and move
//   first (staged E, B), then the region becomes the J tile and all deposit.
//   Two CTAs of 256 threads fit an SM, and each phase's code is short enough
//   for the instruction cache.
// - Particles that leave their cell deposit on other windows; they are listed
//   and deposit one per lane after the pairs, so that no warp runs the wide
//   window for a few lanes.
// - The particles are written to the second buffer in (rank, cell) order:
//   coalesced, and nearly sorted for the next step's reads.
//
// - The components run in a loop over rotated axes: unrolled, the two phases
//   were 130 KB of code and a quarter of all stalls waited for instructions.
//
// Measured (whole step, before -> after): 118 M particles, 1536x256x256 cells,
// 2 per cell 41.3 -> 29.5 ms; 14 M particles, 4 per cell, absorbing layers
// 4.85 -> 2.84 ms; 3.1 M at random places, a quarter leaving their cell each
// step, 1.01 -> 0.78 ms.  With the bodies unrolled the first took 38.6 ms.
// Now issue is active 53 % of cycles; shared memory (loads 1.7 wavefronts
// each) and the latency of the particle loads share the rest.
//
// Exact current: every contribution is an integer product P A, P = round(q w
// jc run 2^kp) below 2^31 with kp per chunk and component, A at 2^30; a node's
// sum over the pair, T = (sum P A + 2^28) >> 29, is added as two 32-bit words,
// hi = T >> 12 and lo = T mod 2^32.  The words give back the exact sum of T:
// it is congruent to lo modulo 2^32 and lies in [2^12 hi, 2^12 (hi + n)) for n
// adds, n < 2^20.  The sum bound B 2^(kp + 1) < 2^42 (B = |q jc| sum |w|)
// keeps hi below 2^30.  The tile sum does not depend on the order of the adds;
// the rounding of P is 2^-32 of the largest |q w jc|, below the 2^-26 or so
// that the FP32 shape factors leave in P itself.
#pragma once

#include "pic_tiled.cuh"

namespace pic {

constexpr int kPushThreads32 = 256;
constexpr int kChunk32 = 3072;  // particles per pass over a tile
constexpr int kRanks32 = 32;    // ranks per cell that are ordered; later ones follow in any order
constexpr unsigned kCross32 = 1u << 31, kStray32 = 1u << 30;

// The shared-memory region in words.  Component d of E, B and J is stored with
// its axes rotated, [i_d][i_e][i_f] with (e, f) the axes after d in cyclic
// order, so that one body serves the three components with the same offsets
// (three unrolled bodies overflow the instruction cache).  E, B: [d][E, B]
// [...]; J: [d][hi, lo][...].  FIXED: tiles of up to 8 cells per axis, strides
// known to the compiler; otherwise any tile.  The fixed strides (12 and 13
// along e, 17 and 12 modulo 32 along d) keep a warp on 4x8 neighbouring cells
// within two wavefronts per access, one for one of the three rotations.
template <bool FIXED>
struct Lay32 {
  int t[3];
  __host__ __device__ explicit Lay32(const Tiles& tl) : t{tl.tx, tl.ty, tl.tz} {}
  // pad = 4: staged fields, 5: J
  __host__ __device__ __forceinline__ int se(int d, int pad) const { return FIXED ? 8 + pad : t[(d + 2) % 3] + pad; }
  __host__ __device__ __forceinline__ int sd(int d, int pad) const {
    return FIXED ? (pad == 4 ? 145 : 172) : (t[(d + 1) % 3] + pad) * se(d, pad);
  }
  __host__ __device__ __forceinline__ int part(int d, int pad) const {
    return FIXED ? (8 + pad) * sd(d, pad) : (t[d] + pad) * sd(d, pad);
  }
  __host__ __device__ __forceinline__ int start(int d, int pad) const { return FIXED ? 2 * d * part(0, pad) : 2 * d * part(d, pad); }
  __host__ __device__ int region(int pad) const { return 6 * part(0, pad); }
  // cell slots: a warp's 32 are 4x8 cells (fixed) or consecutive cells
  __host__ __device__ int words() const { return FIXED ? 2 * t[0] : (t[0] * t[1] * t[2] + 31) / 32; }
  __device__ __forceinline__ int slot(int lx, int ly, int lz) const {
    return FIXED ? lx * 64 + ly * 8 + lz : (lx * t[1] + ly) * t[2] + lz;
  }
  __device__ __forceinline__ void cell(int s, int (&l)[3]) const {
    if (FIXED) {
      l[0] = s >> 6;
      l[1] = (s >> 3) & 7;
      l[2] = s & 7;
    } else {
      l[0] = s / (t[1] * t[2]);
      const int r = s - l[0] * t[1] * t[2];
      l[1] = r / t[2];
      l[2] = r - l[1] * t[2];
    }
  }
};

// Shared memory: the region (staged fields and the ranking's scratch, then J),
// the order list (32-bit entries), the pair list, the list of crossing
// particles, the wrapped grid offsets per axis, and 64 ints of scalars.
struct Smem32 {
  size_t hist, mask, base, order, pair, cross, tab, scal, total;
  template <bool FIXED>
  __host__ __device__ static Smem32 of(const Tiles& tl, const Lay32<FIXED>& L) {
    Smem32 s;
    const size_t w = L.words();
    size_t a = ((size_t)L.region(4) * 4 + 15) / 16 * 16;
    s.hist = a;
    a += 4 * 32 * w;
    s.mask = a;
    a += 4 * kRanks32 * w;
    s.base = a;
    a += (2 * kRanks32 * w + 15) / 16 * 16;
    const size_t j = (size_t)L.region(5) * 4;
    a = ((a > j ? a : j) + 15) / 16 * 16;
    s.order = a;
    a += 4 * (size_t)kChunk32;
    s.pair = a;
    a += 2 * (size_t)kChunk32;
    s.cross = a;
    a += 2 * (size_t)kChunk32;
    s.tab = a;
    a += 4 * (size_t)(tl.tx + tl.ty + tl.tz + 15);
    s.scal = (a + 15) / 16 * 16;
    s.total = s.scal + 4 * 64;
    return s;
  }
};

// Pairs of FP32 values (the two particles of a thread), one instruction for both.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{ .reg .b64 x, y, z, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 z, {%6, %7};"
      " fma.rn.f32x2 w, x, y, z; mov.b64 {%0, %1}, w; }"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{ .reg .b64 x, y, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5};"
      " mul.rn.f32x2 w, x, y; mov.b64 {%0, %1}, w; }"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{ .reg .b64 x, y, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5};"
      " add.rn.f32x2 w, x, y; mov.b64 {%0, %1}, w; }"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 rsqrt2(float2 a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }

// Cubic weights of both particles (see bspline3).
__device__ __forceinline__ void bspline3_2(float2 t, float2 (&w)[4]) {
  const float2 s = add2(dup2(1.0f), neg2(t)), t2 = mul2(t, t), s2 = mul2(s, s), t3 = mul2(t2, t), s3 = mul2(s2, s);
  const float2 sixth = dup2(1.0f / 6.0f), two3 = dup2(2.0f / 3.0f), half = dup2(0.5f);
  w[0] = mul2(s3, sixth);
  w[1] = fma2(t3, half, add2(two3, neg2(t2)));
  w[2] = fma2(s3, half, add2(two3, neg2(s2)));
  w[3] = mul2(t3, sixth);
}

// Node weights (nodes c-1 .. c+2) and half-node weights over c-2 .. c+2 (one
// end zero: the particle's half cell picks the other four).
__device__ __forceinline__ void weights32(float2 o, float2 (&wn)[4], float2 (&wh)[5]) {
  float2 h[4];
  bspline3_2(o, wn);
  const bool lx = o.x < 0.5f, ly = o.y < 0.5f;
  bspline3_2(make_float2(lx ? o.x + 0.5f : o.x - 0.5f, ly ? o.y + 0.5f : o.y - 0.5f), h);
  wh[0] = make_float2(lx ? h[0].x : 0.0f, ly ? h[0].y : 0.0f);
  wh[1] = make_float2(lx ? h[1].x : h[0].x, ly ? h[1].y : h[0].y);
  wh[2] = make_float2(lx ? h[2].x : h[1].x, ly ? h[2].y : h[1].y);
  wh[3] = make_float2(lx ? h[3].x : h[2].x, ly ? h[3].y : h[2].y);
  wh[4] = make_float2(lx ? 0.0f : h[3].x, ly ? 0.0f : h[3].y);
}

// One component for both particles: NA x NB x NC nodes read once, contracted
// along f, then e, then d.
template <int NA, int NB, int NC>
__device__ __forceinline__ float2 gather_pair(const float* __restrict__ s, int sd, int se, const float2* wa,
                                              const float2* wb, const float2* wc) {
  float2 ra;
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    float2 rb;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const float* row = s + a * sd + b * se;
      float f = row[0];
      float2 rc = make_float2(f * wc[0].x, f * wc[0].y);
#pragma unroll
      for (int c = 1; c < NC; ++c) {
        f = row[c];
        rc.x = fmaf(f, wc[c].x, rc.x);
        rc.y = fmaf(f, wc[c].y, rc.y);
      }
      rb = b == 0 ? mul2(rc, wb[0]) : fma2(rc, wb[b], rb);
    }
    ra = a == 0 ? mul2(rb, wa[0]) : fma2(rb, wa[a], ra);
  }
  return ra;
}

// Boris push of both particles in fields E, B: new momenta and 1 / gamma.
__device__ __forceinline__ float2 boris32(float h, const float2 (&E)[3], const float2 (&B)[3], float2 (&u)[3]) {
  const float2 one = dup2(1.0f), hh = dup2(h);
  float2 um[3], tv[3], sv[3], pv[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) um[d] = fma2(hh, E[d], u[d]);
  const float2 hg = mul2(hh, rsqrt2(fma2(um[2], um[2], fma2(um[1], um[1], fma2(um[0], um[0], one)))));  // h / gamma-
#pragma unroll
  for (int d = 0; d < 3; ++d) tv[d] = mul2(hg, B[d]);
  const float2 den = fma2(tv[2], tv[2], fma2(tv[1], tv[1], fma2(tv[0], tv[0], one)));
  const float2 s2 = make_float2(2.0f / den.x, 2.0f / den.y);
#pragma unroll
  for (int d = 0; d < 3; ++d) sv[d] = mul2(s2, tv[d]);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int e = (d + 1) % 3, f = (d + 2) % 3;
    pv[d] = add2(um[d], fma2(um[e], tv[f], neg2(mul2(um[f], tv[e]))));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int e = (d + 1) % 3, f = (d + 2) % 3;
    u[d] = fma2(hh, E[d], add2(um[d], fma2(pv[e], sv[f], neg2(mul2(pv[f], sv[e])))));
  }
  return rsqrt2(fma2(u[2], u[2], fma2(u[1], u[1], fma2(u[0], u[0], one))));
}

// New offset and cell step of one particle along one axis.
__device__ __forceinline__ int step32(float o, float& o1) {
  int k = 0;
  if (o < 0.0f) {
    o += 1.0f;
    k = -1;
  } else if (o >= 1.0f) {
    o -= 1.0f;
    k = 1;
  }
  if (o >= 1.0f) {
    o = 0.0f;
    k += 1;
  }
  o1 = o;
  return k;
}

__device__ __forceinline__ void add_current(unsigned* hi, int lo_off, long long X) {
  const int xh = (int)(X >> 32);
  const unsigned xl = (unsigned)X;
  red_u32(hi, (unsigned)(xh >> 9));                           // T >> 12
  red_u32(hi + lo_off, __funnelshift_r(xl, (unsigned)xh, 29));  // T mod 2^32
}

constexpr float kA30 = 1073741824.0f;  // 2^30
constexpr long long kHalf28 = 1LL << 28;

template <bool FIXED>
__global__ void __launch_bounds__(kPushThreads32, 2)
    k_push32(Geom<float> g, Tiles tl, Fields<float> f, Parts<float> p, Parts<float> pn,
             const int* __restrict__ tstart, int capacity, int* __restrict__ keys, int* __restrict__ cnt_next,
             float h, float q, int origin_after, int xlo, int xhi, unsigned long long* pushed, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (g.dyn) origin_after = g.dyn->origin_after;
  const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int pbeg = min(tstart[t], capacity), pend = min(tstart[t + 1], capacity);
  if (pbeg >= pend) return;
  const Lay32<FIXED> L(tl);
  const Smem32 so = Smem32::of<FIXED>(tl, L);
  float* sF = reinterpret_cast<float*>(smem_raw);
  unsigned* sJ = reinterpret_cast<unsigned*>(smem_raw);
  int* hist = reinterpret_cast<int*>(smem_raw + so.hist);
  unsigned* mask = reinterpret_cast<unsigned*>(smem_raw + so.mask);
  unsigned short* base = reinterpret_cast<unsigned short*>(smem_raw + so.base);
  unsigned* order = reinterpret_cast<unsigned*>(smem_raw + so.order);
  unsigned short* pairB = reinterpret_cast<unsigned short*>(smem_raw + so.pair);
  unsigned short* cross = reinterpret_cast<unsigned short*>(smem_raw + so.cross);
  int* tabx = reinterpret_cast<int*>(smem_raw + so.tab);
  int* taby = tabx + tl.tx + 5;
  int* tabz = taby + tl.ty + 5;
  // scalars: [0] tail count, [1] crossing count, [2] sum |w|, [3] max |w|
  // (bits), [4, 7) kp, [8, 16) scan partials, [16, 33) first pair of a round,
  // [33] ranked particles, [34, 50) first position of a round's first particles
  int* sc = reinterpret_cast<int*>(smem_raw + so.scal);
  const int W = L.words();
  const int tzi = t % tl.ntz, rest = t / tl.ntz;
  const int x0 = (rest / tl.nty) * tl.tx, y0 = (rest % tl.nty) * tl.ty, z0 = tzi * tl.tz;

  // wrapped grid offsets of the staged cells (origin tile - 2; J reaches one
  // cell further than E, B)
  for (int i = tid; i < tl.tx + tl.ty + tl.tz + 15; i += kPushThreads32) {
    int v;
    if (i < tl.tx + 5)
      v = wrapi(x0 - 2 + i, g.nx) * g.nyz;
    else if (i < tl.tx + tl.ty + 10)
      v = wrapi(y0 - 2 + i - (tl.tx + 5), g.ny) * g.nz;
    else
      v = wrapi(z0 - 2 + i - (tl.tx + tl.ty + 10), g.nz);
    tabx[i] = v;
  }
  const int ntile = pend - pbeg;
  if (tid == 0) {
    atomicAdd(pushed, (unsigned long long)ntile);
    if (ntile >= (1 << 20)) atomicOr(err, 16);
  }
  const int npass = (ntile + kChunk32 - 1) / kChunk32, per_pass = (ntile + npass - 1) / npass;
  const float dtd[3] = {g.dt / g.dx, g.dt / g.dy, g.dt / g.dz};
  int own = 0;

  for (int ch0 = 0; ch0 < ntile; ch0 += per_pass) {
    const int nch = min(per_pass, ntile - ch0), c0 = pbeg + ch0;
    for (int i = tid; i < 32 * W; i += kPushThreads32) hist[i] = 0;
    for (int i = tid; i < kRanks32 * W; i += kPushThreads32) mask[i] = 0u;
    if (tid < 64) sc[tid] = 0;
    __syncthreads();

    // stage E, B: a half warp per (x, y) row, the lanes along z
    {
      const int SY = tl.ty + 4, rows = (tl.tx + 4) * SY, SZ = tl.tz + 4;
      for (int r = tid >> 4; r < rows; r += kPushThreads32 / 16) {
        const int lx = r / SY, ly = r - lx * SY;
        const int gi0 = tabx[lx] + taby[ly];
        for (int lz = tid & 15; lz < SZ; lz += 16) {
          const int gi = gi0 + tabz[lz];
          const int i3[3] = {lx, ly, lz};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const float* dst = sF + L.start(d, 4) + i3[d] * L.sd(d, 4) + i3[(d + 1) % 3] * L.se(d, 4) + i3[(d + 2) % 3];
            const unsigned a = (unsigned)__cvta_generic_to_shared(dst);
            const unsigned b = a + 4u * (unsigned)L.part(d, 4);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a), "l"(f.c[EX + d] + gi) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(b), "l"(f.c[BX + d] + gi) : "memory");
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }

    // rank the chunk's particles per cell; sum and maximum of |w|
    constexpr int kPer = kChunk32 / kPushThreads32;
    int sr[kPer];
    float ws = 0.0f, wm = 0.0f;
    const float inv_nyz = 1.0f / (float)g.nyz, inv_nz = 1.0f / (float)g.nz;
#pragma unroll
    for (int it = 0; it < kPer; ++it) {
      const int k = it * kPushThreads32 + tid;
      sr[it] = -1;
      if (k < nch) {
        const int cell = p.cell[c0 + k];
        const float wa = fabsf(p.w[c0 + k]);
        ws += wa;
        wm = fmaxf(wm, wa);
        // cell - (tile corner) split by quotient estimates, then checked exactly
        const int rel = cell - x0 * g.nyz - y0 * g.nz - z0;
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
          sr[it] = s | (atomicAdd(hist + s, 1) << 12);
        } else {  // never expected: keeps every index in range
          atomicOr(err, 4);
          sr[it] = -2;
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ws += __shfl_down_sync(0xffffffffu, ws, o);
      wm = fmaxf(wm, __shfl_down_sync(0xffffffffu, wm, o));
    }
    if (lane == 0) {
      atomicAdd(reinterpret_cast<float*>(sc + 2), ws);
      atomicMax(sc + 3, __float_as_int(wm));
    }
    __syncthreads();

    // occupancy of every rank: bit of a slot set in mask[r][word] if the cell
    // holds more than r particles
    for (int i = tid; i < 32 * W; i += kPushThreads32) {
      const int n = min(hist[i], kRanks32);
      for (int r = 0;; ++r) {
        const unsigned m = __ballot_sync(0xffffffffu, n > r);
        if (!m) break;
        if (lane == 0) mask[r * W + (i >> 5)] = m;
      }
    }
    if (tid < 3) {
      // kp: |P| 2^kp < 2^31 for P <= 0.76 |q| max w jc, and B 2^(kp + 1) < 2^42
      const float jcc = tid == 0 ? g.dt * g.dy * g.dz : (tid == 1 ? g.dt * g.dx * g.dz : g.dt * g.dx * g.dy);
      const float P = 0.76f * fabsf(q) * __int_as_float(sc[3]) / jcc;
      const float B = 1.001f * fabsf(q) * __int_as_float(sc[2]) / jcc;
      const int ep = ((__float_as_int(P) >> 23) & 255) - 127, eb = ((__float_as_int(B) >> 23) & 255) - 127;
      sc[4 + tid] = B > 0.0f ? max(min(min(30 - ep, 40 - eb), 120), -120) : 0;
    }
    __syncthreads();
    // exclusive scan of the population counts over (rank, word)
    {
      const int n = kRanks32 * W, per = (n + kPushThreads32 - 1) / kPushThreads32;
      const int b = min(tid * per, n), e = min(b + per, n);
      int s = 0;
      for (int i = b; i < e; ++i) s += __popc(mask[i]);
      int incl = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) sc[8 + (tid >> 5)] = incl;
      __syncthreads();
      int run = incl - s;
      for (int k = 0; k < (tid >> 5); ++k) run += sc[8 + k];
      for (int i = b; i < e; ++i) {
        base[i] = (unsigned short)run;
        run += __popc(mask[i]);
      }
      if (tid == kPushThreads32 - 1) sc[33] = run;
    }
    __syncthreads();
    // pairs of a round: as many as the round's first particles
    if (tid < 32) {
      const int r = 2 * min(lane, kRanks32 / 2 - 1);
      const int first = base[r * W], next = base[(r + 1) * W];
      const int n = lane < kRanks32 / 2 ? next - first : 0;
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane <= kRanks32 / 2) sc[16 + lane] = incl - n;
      if (lane < kRanks32 / 2) sc[34 + lane] = first;
    }
    const int ranked = sc[33];
#pragma unroll
    for (int it = 0; it < kPer; ++it) {
      const int k = it * kPushThreads32 + tid;
      if (k < nch) {
        const int v = sr[it];
        const int s = v & 4095, r = v >> 12;
        int pos;
        unsigned e = (unsigned)k | ((unsigned)s << 12);
        if (v == -2) e = (unsigned)k | kStray32;
        if (v != -2 && r < kRanks32)
          pos = base[r * W + (s >> 5)] + __popc(mask[r * W + (s >> 5)] & ((1u << (s & 31)) - 1u));
        else
          pos = ranked + atomicAdd(sc, 1);
        order[pos] = e;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    const int nround = sc[16 + kRanks32 / 2];       // pairs of the ordered ranks
    const int nitem = nround + (nch - ranked);      // the rest goes one by one
    // ---- gather, push, move ----
    int round = 0;
    for (int i0 = 0; i0 < nitem; i0 += kPushThreads32) {
      const int i = i0 + tid;
      bool have[2] = {i < nitem, false};
      int pos[2] = {0, 0};
      if (have[0]) {
        if (i < nround) {
          while (i >= sc[17 + round]) ++round;
          pos[0] = sc[34 + round] + i - sc[16 + round];
        } else {
          pos[0] = ranked + i - nround;
        }
      }
      unsigned ent[2];
      ent[0] = have[0] ? order[pos[0]] : kStray32;
      if (have[0] && (ent[0] & kStray32)) {  // dropped with the error bit set
        keys[c0 + pos[0]] = -1;
        order[pos[0]] = ent[0] | kCross32;
      }
      have[0] = have[0] && !(ent[0] & kStray32);
      const int s = (ent[0] >> 12) & 4095;
      if (have[0] && i < nround) {
        const int w = (2 * round + 1) * W + (s >> 5);
        const unsigned m = mask[w];
        have[1] = (m >> (s & 31)) & 1u;
        pos[1] = base[w] + __popc(m & ((1u << (s & 31)) - 1u));
      }
      if (i < nitem) pairB[i] = have[1] ? (unsigned short)pos[1] : (unsigned short)0xffff;
      ent[1] = have[1] ? order[pos[1]] : ent[0];
      int key[2] = {-2, -2};
      if (have[0]) {
        int l[3];
        L.cell(s, l);
        const int idx[2] = {c0 + (int)(ent[0] & 4095), c0 + (int)(ent[1] & 4095)};
        float2 u[3], E[3], B[3];
        {
          float2 wn[3][4], wh[3][5];
#pragma unroll
          for (int d = 0; d < 3; ++d) weights32(make_float2(p.o[d][idx[0]], p.o[d][idx[1]]), wn[d], wh[d]);
          int r[3] = {l[0], l[1], l[2]};
#pragma unroll 1
          for (int d = 0; d < 3; ++d) {  // axes 0, 1, 2 of the arrays: d, e, f
            const int sd = L.sd(d, 4), se = L.se(d, 4);
            // node-centred axes start at c-1, half-staggered ones at c-2
            const float* b = sF + L.start(d, 4) + r[0] * sd + r[1] * se + r[2];
            const float2 e = gather_pair<5, 4, 4>(b + se + 1, sd, se, wh[0], wn[1], wn[2]);
            const float2 m = gather_pair<4, 5, 5>(b + L.part(d, 4) + sd, sd, se, wn[0], wh[1], wh[2]);
            E[0] = E[1], E[1] = E[2], E[2] = e;
            B[0] = B[1], B[1] = B[2], B[2] = m;
            const int r0 = r[0];
            r[0] = r[1], r[1] = r[2], r[2] = r0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 v = wn[0][k];
              wn[0][k] = wn[1][k], wn[1][k] = wn[2][k], wn[2][k] = v;
            }
#pragma unroll
            for (int k = 0; k < 5; ++k) {
              const float2 v = wh[0][k];
              wh[0][k] = wh[1][k], wh[1][k] = wh[2][k], wh[2][k] = v;
            }
          }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d] = make_float2(p.u[d][idx[0]], p.u[d][idx[1]]);
        const float2 ig = boris32(h, E, B, u);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (k == 1 && !have[1]) break;
          const float igk = k ? ig.y : ig.x;
          float uk[3] = {k ? u[0].y : u[0].x, k ? u[1].y : u[1].x, k ? u[2].y : u[2].x};
          const bool good = igk > 0.0f;
          if (!good) {  // a non-finite momentum: reported; absorbed without moving or depositing
            atomicOr(err, 8);
            uk[0] = uk[1] = uk[2] = 0.0f;
          }
          int dc[3];
          const int dst = c0 + pos[k];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const float o = p.o[d][idx[k]];
            float o1;
            dc[d] = step32(good ? o + dtd[d] * uk[d] * igk : o, o1);
            pn.o[d][dst] = o1;
            pn.u[d][dst] = uk[d];
          }
          pn.w[dst] = p.w[idx[k]];
          if (pn.id) pn.id[dst] = p.id[idx[k]];
          // the new cell and its tile: a move is at most one cell, across the grid's end to the first or last tile
          int n0 = x0 + l[0] + dc[0], n1 = y0 + l[1] + dc[1], n2 = z0 + l[2] + dc[2];
          key[k] = t;
          if (dc[0] | dc[1] | dc[2]) {
            n0 = wrapi(n0, g.nx), n1 = wrapi(n1, g.ny), n2 = wrapi(n2, g.nz);
            if ((unsigned)(n0 - x0) >= (unsigned)tl.tx || (unsigned)(n1 - y0) >= (unsigned)tl.ty ||
                (unsigned)(n2 - z0) >= (unsigned)tl.tz)
              key[k] = tile_of(g, tl, n0, n1, n2);
            order[pos[k]] = ent[k] | kCross32 | ((unsigned)(dc[0] + 1) << 24) | ((unsigned)(dc[1] + 1) << 26) |
                            ((unsigned)(dc[2] + 1) << 28);
            cross[atomicAdd(sc + 1, 1)] = (unsigned short)pos[k];
          }
          pn.cell[dst] = (n0 * g.ny + n1) * g.nz + n2;
          if (!g.periodic_x) {
            int rel = n0 - origin_after;
            if (rel < 0) rel += g.nx;
            if (rel < xlo || rel > xhi) key[k] = -1;
          }
          // absorbing layers: a particle that leaves the y, z cells [L, n - L) is absorbed
          if (g.pml && (n1 < g.pml || n1 >= g.ny - g.pml || n2 < g.pml || n2 >= g.nz - g.pml)) key[k] = -1;
          if (!good) {
            key[k] = -1;
            order[pos[k]] = ent[k] | kCross32;
          }
          keys[dst] = key[k];
          if (key[k] == t) own += 1;
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int kk = key[k] == t ? -2 : key[k];
        if (__any_sync(0xffffffffu, kk >= 0)) warp_count(cnt_next, kk, false, nullptr);
      }
    }
    __syncthreads();

    // ---- the region becomes the J tile ----
    {
      int4* z = reinterpret_cast<int4*>(smem_raw);
      const int n = (int)(so.order / 16);
      for (int i = tid; i < n; i += kPushThreads32) z[i] = make_int4(0, 0, 0, 0);
    }
    __syncthreads();
    const float third = 1.0f / 3.0f;
    const float jcc[3] = {g.dt * g.dy * g.dz, g.dt * g.dx * g.dz, g.dt * g.dx * g.dy};
    round = 0;
    for (int i = tid; i < nitem; i += kPushThreads32) {
      int posA;
      if (i < nround) {
        while (i >= sc[17 + round]) ++round;
        posA = sc[34 + round] + i - sc[16 + round];
      } else {
        posA = ranked + i - nround;
      }
      const int pb = pairB[i];
      const int pos[2] = {posA, pb == 0xffff ? posA : pb};
      const unsigned ent[2] = {order[pos[0]], order[pos[1]]};
      const bool dep[2] = {!(ent[0] & kCross32), pb != 0xffff && !(ent[1] & kCross32)};
      if (!(dep[0] || dep[1])) continue;
      int r[3];
      L.cell((ent[0] >> 12) & 4095, r);
      float2 S[3][4], D[3][4], qw;
      {
        const int i0 = c0 + (int)(ent[0] & 4095), i1 = c0 + (int)(ent[1] & 4095), d0 = c0 + pos[0], d1 = c0 + pos[1];
        qw = make_float2(dep[0] ? q * p.w[i0] : 0.0f, dep[1] ? q * p.w[i1] : 0.0f);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float2 a = make_float2(p.o[d][i0], p.o[d][i1]);
          const float2 b = make_float2(dep[0] ? pn.o[d][d0] : a.x, dep[1] ? pn.o[d][d1] : a.y);
          float2 w1[4];
          bspline3_2(a, S[d]);
          bspline3_2(b, w1);
#pragma unroll
          for (int k = 0; k < 4; ++k) D[d][k] = add2(w1[k], neg2(S[d][k]));
        }
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {  // axes 0, 1, 2 of the arrays: d, e, f
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + (r[0] + 1) * sd + (r[1] + 1) * se + r[2] + 1;  // nodes c-1 .. c+2
        int P[2][3];
        {
          const float scale = __int_as_float((127 + sc[4 + d]) << 23);
          const float jc = -1.0f / (d == 0 ? jcc[0] : (d == 1 ? jcc[1] : jcc[2]));
          const float2 c = mul2(mul2(dup2(jc), qw), dup2(scale));
          float2 run = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            run = add2(run, D[0][m]);
            const float2 v = mul2(c, run);
            P[0][m] = __float2int_rn(v.x);
            P[1][m] = __float2int_rn(v.y);
          }
        }
        // A(b, c) = S_e (S_f + D_f / 2) + D_e (S_f / 2 + D_f / 3)
        float2 ak[4], bk[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          ak[m] = mul2(dup2(kA30), fma2(dup2(0.5f), D[2][m], S[2][m]));
          bk[m] = mul2(dup2(kA30), fma2(dup2(third), D[2][m], mul2(dup2(0.5f), S[2][m])));
        }
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float2 A = fma2(D[1][b], bk[c], mul2(S[1][b], ak[c]));
            const int A0 = __float2int_rn(A.x), A1 = __float2int_rn(A.y);
#pragma unroll
            for (int m = 0; m < 3; ++m)
              add_current(j + m * sd + b * se + c, lo, kHalf28 + (long long)P[0][m] * A0 + (long long)P[1][m] * A1);
          }
        const int r0 = r[0];
        r[0] = r[1], r[1] = r[2], r[2] = r0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 v = S[0][k], w = D[0][k];
          S[0][k] = S[1][k], S[1][k] = S[2][k], S[2][k] = v;
          D[0][k] = D[1][k], D[1][k] = D[2][k], D[2][k] = w;
        }
      }
    }
    // particles that left their cell: 5-node windows where they moved
    const int ncross = sc[1];
    for (int i = tid; i < ncross; i += kPushThreads32) {
      const int pos = cross[i];
      const unsigned e = order[pos];
      int r[3], n[3];
      L.cell((e >> 12) & 4095, r);
      const int idx = c0 + (int)(e & 4095), dst = c0 + pos;
      const float qw = q * p.w[idx];
      float S[3][5], D[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int dc = (int)((e >> (24 + 2 * d)) & 3u) - 1;
        float wn[4], w1[4];
        bspline3(p.o[d][idx], wn);
        bspline3(pn.o[d][dst], w1);
        const int p0 = dc < 0 ? 1 : 0, p1 = dc > 0 ? 1 : 0;
        r[d] += 1 - p0;
        n[d] = dc != 0 ? 5 : 4;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const float a0 = p0 ? (m > 0 ? wn[m > 0 ? m - 1 : 0] : 0.0f) : (m < 4 ? wn[m < 4 ? m : 3] : 0.0f);
          const float a1 = p1 ? (m > 0 ? w1[m > 0 ? m - 1 : 0] : 0.0f) : (m < 4 ? w1[m < 4 ? m : 3] : 0.0f);
          S[d][m] = a0;
          D[d][m] = a1 - a0;
        }
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + r[0] * sd + r[1] * se + r[2];
        int P[4];
        {
          const float scale = __int_as_float((127 + sc[4 + d]) << 23);
          const float c = -1.0f / (d == 0 ? jcc[0] : (d == 1 ? jcc[1] : jcc[2])) * qw * scale;
          float run = 0.0f;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            run += D[0][m];
            P[m] = __float2int_rn(c * run);
          }
        }
        float ak[5], bk[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          ak[m] = kA30 * (S[2][m] + 0.5f * D[2][m]);
          bk[m] = kA30 * (0.5f * S[2][m] + third * D[2][m]);
        }
#pragma unroll
        for (int b = 0; b < 5; ++b)
          if (b < n[1]) {
#pragma unroll
            for (int c = 0; c < 5; ++c)
              if (c < n[2]) {
                const int A = __float2int_rn(S[1][b] * ak[c] + D[1][b] * bk[c]);
#pragma unroll
                for (int m = 0; m < 4; ++m)
                  if (m < n[0] - 1) add_current(j + m * sd + b * se + c, lo, kHalf28 + (long long)P[m] * A);
              }
          }
        const int r0 = r[0], n0 = n[0];
        r[0] = r[1], r[1] = r[2], r[2] = r0;
        n[0] = n[1], n[1] = n[2], n[2] = n0;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const float v = S[0][k], w = D[0][k];
          S[0][k] = S[1][k], S[1][k] = S[2][k], S[2][k] = v;
          D[0][k] = D[1][k], D[1][k] = D[2][k], D[2][k] = w;
        }
      }
    }
    __syncthreads();

    // flush: a half warp per (x, y) row, the lanes along z
    {
      const int NY = tl.ty + 5, rows = (tl.tx + 5) * NY, NZ = tl.tz + 5;
      for (int r = tid >> 4; r < rows; r += kPushThreads32 / 16) {
        const int lx = r / NY, ly = r - lx * NY;
        const int gi0 = tabx[lx] + taby[ly];
        for (int lz = tid & 15; lz < NZ; lz += 16) {
          const int i3[3] = {lx, ly, lz};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const unsigned* w = sJ + L.start(d, 5) + i3[d] * L.sd(d, 5) + i3[(d + 1) % 3] * L.se(d, 5) + i3[(d + 2) % 3];
            const unsigned hi = w[0], lo = w[L.part(d, 5)];
            if (hi | lo) {
              // T = top 2^21 + low, both exact as floats: one rounding
              const long long T = (long long)(int)hi * 4096 + (long long)(lo - (hi << 12));
              const float v = fmaf((float)(int)(T >> 21), 2097152.0f, (float)(int)(T & 0x1fffff));
              atomicAdd(f.c[JX + d] + gi0 + tabz[lz], v * __int_as_float((126 - sc[4 + d]) << 23));  // 2^-(kp + 1)
            }
          }
        }
      }
    }
    __syncthreads();
  }
  own = __reduce_add_sync(0xffffffffu, own);
  if (lane == 0 && own) atomicAdd(cnt_next + t, own);
}

}  // namespace pic
