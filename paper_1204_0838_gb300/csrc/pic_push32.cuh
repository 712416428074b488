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
//   Each phase's code is short enough for the instruction cache.
// - Particles that leave their cell deposit on other windows; they are listed
//   and deposit one per lane after the pairs, so that no warp runs the wide
//   window for a few lanes.
// - The particles are written to the second buffer in (rank, cell) order:
//   coalesced, and nearly sorted for the next step's reads.
//
// - The components run in a loop over rotated axes: unrolled, the two phases
//   were 130 KB of code and a quarter of all stalls waited for instructions.
//
// - Three CTAs of 256 threads per SM at 80 registers: the weights are formed
//   again for every rotation instead of kept; two particles' arithmetic goes in
//   packed FP32 instructions.
//
// Measured (whole step, the one-pass kernel -> this one): 118 M particles,
// 1536x256x256 cells, 2 per cell 41.3 -> 26.1 ms; 14 M particles, 4 per cell,
// absorbing layers 4.85 -> 2.51 ms; 3.1 M at random places, a quarter leaving
// their cell each step, 1.01 -> 0.72 ms.  With the bodies unrolled the first took
// 38.6 ms, with two CTAs at 128 registers 27.6.  In a run's state, 2 per cell: 3,370
// instructions per 32 particles, issued 49 % of the time, the shared-memory pipe 76 %
// busy; waits at barriers (uneven last rounds of a tile) and for shared memory are the
// largest stalls.
//
// Current: sums of integers at 2^s per tile and component, with s the largest
// for which B 2^s < 2^42, B = |q jc| sum |w|.  A contribution is a product of
// two rounded integers, P = q w jc run at 2^kp, below 2^31, and A at 2^31; a
// pair's P A are added exactly and rounded once, T = sum P A >> (kp + 31 - s),
// and T is added as two 32-bit words, hi = T >> 12 and lo = T mod 2^32.  The
// words give back the exact sum of T: it is congruent to lo modulo 2^32 and
// lies in [2^12 hi, 2^12 (hi + n)) for n adds, n < 2^20; hi stays below 2^31.
// So the sum does not depend on the order of the adds.  A contribution is
// rounded by 2^-42 of B, and P, if less than that, by
// - 2^-31 of the tile's largest |q w jc| for particles within 8 of the largest
//   weight, which share kp: at most 2^-28 of their own |q w jc|, below the 2^-26
//   or so that the FP32 shape factors leave in P itself;
// - 2^-31 of its own |q w jc| for a lighter particle or one that left its cell:
//   these deposit one per lane, with a kp of their own.  (With one kp for all, the
//   current of particles at 1e-4 of the largest weight was off by 1e-4 of itself,
//   of those at 1e-6 by 1e-2.  A step of 1.6 M particles takes 414 us with equal
//   weights, 493 with one in a hundred a hundred times heavier, so that nearly all
//   others are light.)
#pragma once

#include "pic_push.cuh"

namespace pic {

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
__device__ __forceinline__ float2 rsqrt2(float2 a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }

// Cubic B-spline weights of the nodes c-1 .. c+2 for an offset t (see bspline3).
// 2/3 is carried as a value and its remainder: rounded up alone, the weights of an
// axis would sum to 4e-8 above one, and the current to twice that.
__device__ __forceinline__ void spline32(float2 t, float2 (&w)[4]) {
  constexpr float hi = 2.0f / 3.0f, lo = (float)(2.0 / 3.0 - (double)hi), sixth = 1.0f / 6.0f;
  const float2 s = fma2(t, dup2(-1.0f), dup2(1.0f)), t2 = mul2(t, t), s2 = mul2(s, s), t3 = mul2(t2, t), s3 = mul2(s2, s);
  w[0] = mul2(s3, dup2(sixth));
  w[1] = add2(fma2(t2, dup2(-1.0f), dup2(hi)), fma2(t3, dup2(0.5f), dup2(lo)));
  w[2] = add2(fma2(s2, dup2(-1.0f), dup2(hi)), fma2(s3, dup2(0.5f), dup2(lo)));
  w[3] = mul2(t3, dup2(sixth));
}

// Half-node weights over c-2 .. c+2 (one end zero: the particle's half cell
// picks the other four).
__device__ __forceinline__ void half_weights32(float2 o, float2 (&wh)[5]) {
  float2 h[4];
  const bool lx = o.x < 0.5f, ly = o.y < 0.5f;
  spline32(make_float2(lx ? o.x + 0.5f : o.x - 0.5f, ly ? o.y + 0.5f : o.y - 0.5f), h);
  wh[0] = make_float2(lx ? h[0].x : 0.0f, ly ? h[0].y : 0.0f);
  wh[1] = make_float2(lx ? h[1].x : h[0].x, ly ? h[1].y : h[0].y);
  wh[2] = make_float2(lx ? h[2].x : h[1].x, ly ? h[2].y : h[1].y);
  wh[3] = make_float2(lx ? h[3].x : h[2].x, ly ? h[3].y : h[2].y);
  wh[4] = make_float2(lx ? 0.0f : h[3].x, ly ? 0.0f : h[3].y);
}

// Shape factors of both particles at an axis's old offsets, and their change.
__device__ __forceinline__ void shapes32(float2 o0, float2 o1, float2 (&S)[4], float2 (&D)[4]) {
  float2 w1[4];
  spline32(o0, S);
  spline32(o1, w1);
#pragma unroll
  for (int k = 0; k < 4; ++k) D[k] = fma2(S[k], dup2(-1.0f), w1[k]);
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
      float2 rc = mul2(dup2(row[0]), wc[0]);  // a value for both halves costs no move
#pragma unroll
      for (int c = 1; c < NC; ++c) rc = fma2(dup2(row[c]), wc[c], rc);
      rb = b == 0 ? mul2(rc, wb[0]) : fma2(rc, wb[b], rb);
    }
    ra = a == 0 ? mul2(rb, wa[0]) : fma2(rb, wa[a], ra);
  }
  return ra;
}

// Boris push of both particles in fields E, B: new momenta and 1 / gamma.
__device__ __forceinline__ float2 boris32(float h, const float2 (&E)[3], const float2 (&B)[3], float2 (&u)[3]) {
  const float2 one = dup2(1.0f), hh = dup2(h);
  float2 um[3], tv[3], tn[3], pv[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) um[d] = fma2(hh, E[d], u[d]);
  const float2 hg = mul2(hh, rsqrt2(fma2(um[2], um[2], fma2(um[1], um[1], fma2(um[0], um[0], one)))));  // h / gamma-
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    tv[d] = mul2(hg, B[d]);
    tn[d] = mul2(tv[d], dup2(-1.0f));
  }
  const float2 den = fma2(tv[2], tv[2], fma2(tv[1], tv[1], fma2(tv[0], tv[0], one)));
  const float2 s2 = make_float2(2.0f / den.x, 2.0f / den.y);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int e = (d + 1) % 3, f = (d + 2) % 3;
    pv[d] = add2(um[d], fma2(um[e], tv[f], mul2(um[f], tn[e])));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int e = (d + 1) % 3, f = (d + 2) % 3;
    u[d] = fma2(hh, E[d], fma2(s2, fma2(pv[e], tv[f], mul2(pv[f], tn[e])), um[d]));
  }
  return rsqrt2(fma2(u[2], u[2], fma2(u[1], u[1], fma2(u[0], u[0], one))));
}

// The push of one particle with the fields of its own 4x4x4 windows (both halves the
// same particle).  Returns 1 / gamma.
template <bool FIXED>
__device__ __forceinline__ float push_own32(const float* sF, const PushLayout<float, FIXED>& L, const int (&l)[3], float h,
                                            float2 (&o)[3], float2 (&u)[3]) {
  float2 E[3], B[3];
  int r[3] = {l[0], l[1], l[2]};
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    const int sd = L.sd(d, 4), se = L.se(d, 4);
    float2 wn[3][4], wh[3][4];
    int hi[3];  // half-node windows start at c-2 or, from half a cell on, at c-1
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      hi[a] = o[a].x < 0.5f ? 0 : 1;
      spline32(o[a], wn[a]);
      spline32(add2(o[a], dup2(hi[a] ? -0.5f : 0.5f)), wh[a]);
    }
    const float* b = sF + L.start(d, 4) + r[0] * sd + r[1] * se + r[2];
    E[0] = E[1], E[1] = E[2];
    B[0] = B[1], B[1] = B[2];
    E[2] = gather_pair<4, 4, 4>(b + hi[0] * sd + se + 1, sd, se, wh[0], wn[1], wn[2]);
    B[2] = gather_pair<4, 4, 4>(b + L.part(d, 4) + sd + hi[1] * se + hi[2], sd, se, wn[0], wh[1], wh[2]);
    const int r0 = r[0];
    r[0] = r[1], r[1] = r[2], r[2] = r0;
    const float2 t = o[0];
    o[0] = o[1], o[1] = o[2], o[2] = t;
  }
  return boris32(h, E, B, u).x;
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

// Add T = X >> sh, 20 <= sh <= 31 (X holds the rounding half already).
__device__ __forceinline__ void add_current(unsigned* hi, int lo_off, long long X, int sh) {
  const int xh = (int)(X >> 32);
  const unsigned xl = (unsigned)X;
  red_u32(hi, (unsigned)(xh >> (sh - 20)));                   // T >> 12
  red_u32(hi + lo_off, __funnelshift_r(xl, (unsigned)xh, sh));  // T mod 2^32
}

constexpr float kA31 = 2147483648.0f;  // 2^31; A is at most 4/9
constexpr float kLight = 0.125f;       // of the largest weight: below it a particle has its own kp

template <bool FIXED>
__global__ void __launch_bounds__(kPushThreads, 3)
    k_push32(Geom<float> g, Tiles tl, Fields<float> f, Parts<float> p, Parts<float> pn,
             const int* __restrict__ tstart, int capacity, int* __restrict__ keys, int* __restrict__ cnt_next,
             PushCoef<float> pc, int origin_after, int xlo, int xhi, unsigned long long* pushed, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (g.dyn) origin_after = g.dyn->origin_after;
  const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int pbeg = min(tstart[t], capacity), pend = min(tstart[t + 1], capacity);
  if (pbeg >= pend) return;
  const PushLayout<float, FIXED> L(tl);
  const PushTile P = push_tile<float, FIXED>(smem_raw, g, tl, t);
  const PushSmem so = PushSmem::of<float, FIXED>(tl);
  float* sF = reinterpret_cast<float*>(smem_raw);
  unsigned* sJ = reinterpret_cast<unsigned*>(smem_raw);
  unsigned short* pairB = reinterpret_cast<unsigned short*>(smem_raw + so.pair);
  unsigned* order = P.order;
  int* sc = P.sc;
  const int W = L.words();
  const int ntile = pend - pbeg;
  if (tid == 0) {
    atomicAdd(pushed, (unsigned long long)ntile);
    if (ntile >= (1 << 20)) atomicOr(err, 16);
  }
  const int npass = (ntile + kChunk - 1) / kChunk;
  int own = 0;

  for (int ps = 0; ps < npass; ++ps) {
    const Pass pass(ps, npass, ntile);
    const int nch = pass.n, c0 = pbeg + pass.begin;
    rank_clear(P, W);
    __syncthreads();

    // stage E, B: a half warp per (x, y) row, the lanes along z
    if (ps == 0) {
      const int SX = tl.tx + 4, SZ = tl.tz + 4;
      for (RowWalk r(tl.ty + 4); r.lx < SX; r.next()) {
        const int lx = r.lx, ly = r.ly;
        const int gi0 = P.tabx[lx] + P.taby[ly];
        for (int lz = tid & 15; lz < SZ; lz += 16) {
          const int gi = gi0 + P.tabz[lz];
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

    // rank the pass's particles per cell; sum and maximum of |w| over the tile
    int sr[kPerThread];
    rank_count(P, L, g, tl, p.cell, c0, nch, sr, err);
    if (ps == 0) {
      float ws = 0.0f, wm = 0.0f;
      for (int k = tid; k < ntile; k += kPushThreads) {
        const float wa = fabsf(p.w[pbeg + k]);
        ws += wa;
        wm = fmaxf(wm, wa);
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
    }
    __syncthreads();
    rank_masks(P, W);
    if (ps == 0 && tid < 3) {
      // s: B 2^s < 2^42; kp: |P| 2^kp < 2^31 for P <= 0.76 |q| max w jc, no finer
      // than s.  B > Pm, so that 20 <= kp + 31 - s <= 31.
      const float jc = fabsf(pc.q * (tid == 0 ? pc.jc[0] : (tid == 1 ? pc.jc[1] : pc.jc[2])));
      const float wm = __int_as_float(sc[3]);
      const float Pm = 0.76f * jc * wm, B = 1.001f * jc * __int_as_float(sc[2]);
      const int ep = ((__float_as_int(Pm) >> 23) & 255) - 127, eb = ((__float_as_int(B) >> 23) & 255) - 127;
      const int s = B > 0.0f ? min(41 - eb, 120) : 0;
      const int kp = B > 0.0f ? max(min(30 - ep, s), s - 11) : 0;
      sc[4 + tid] = s;
      sc[50 + tid] = kp;
      if (kp < s) atomicMax(sc + 53, __float_as_int(kLight * wm));
    }
    __syncthreads();
    rank_order(P, W, nch, sr);
    // pairs of ranks 2k, 2k + 1: as many as particles of rank 2k
    if (tid < 32) {
      const int r = 2 * min(lane, kRanks / 2 - 1);
      const int first = P.base[r * W], next = P.base[(r + 1) * W];
      const int n = lane < kRanks / 2 ? next - first : 0;
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane <= kRanks / 2) sc[16 + lane] = incl - n;
      if (lane < kRanks / 2) sc[34 + lane] = first;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    const int ranked = sc[33];
    const int nround = sc[16 + kRanks / 2];       // pairs of the ordered ranks
    const int nitem = nround + (nch - ranked);      // the rest goes one by one
    // Move a particle with momentum u and 1 / gamma; returns its destination tile.
    auto finish = [&](const int(&l)[3], int idx, int pos, unsigned ent, const float(&u)[3], float ig, bool good) {
      int dc[3];
      const int dst = c0 + pos;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float o = p.o[d][idx];
        float o1;
        dc[d] = step32(good ? o + pc.dtd[d] * u[d] * ig : o, o1);
        pn.o[d][dst] = o1;
        pn.u[d][dst] = u[d];
      }
      const float w = p.w[idx];
      pn.w[dst] = w;
      if (pn.id) pn.id[dst] = p.id[idx];
      return place_moved(P, g, tl, t, l, dc, good, good && fabsf(w) < __int_as_float(sc[53]), origin_after, xlo, xhi, pos, ent,
                         pn.cell + dst, keys + dst);
    };
    // ---- gather, push, move ----
    int round = 0;
    for (int i0 = 0; i0 < nitem; i0 += kPushThreads) {
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
      ent[0] = have[0] ? order[pos[0]] : kStray;
      if (have[0] && (ent[0] & kStray)) {  // dropped with the error bit set
        keys[c0 + pos[0]] = -1;
        order[pos[0]] = ent[0] | kCross;
      }
      have[0] = have[0] && !(ent[0] & kStray);
      const int s = (ent[0] >> 12) & 4095;
      if (have[0] && i < nround) {
        have[1] = (P.mask[(2 * round + 1) * W + (s >> 5)] >> (s & 31)) & 1u;
        pos[1] = P.position(W, 2 * round + 1, s);
      }
      if (i < nitem) pairB[i] = have[1] ? (unsigned short)pos[1] : (unsigned short)0xffff;
      ent[1] = have[1] ? order[pos[1]] : ent[0];
      int key[2] = {-2, -2};
      if (have[0]) {
        int l[3];
        L.cell(s, l);
        const int idx[2] = {c0 + (int)(ent[0] & 4095), c0 + (int)(ent[1] & 4095)};
        float2 u[3], E[3], B[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {  // for after the gather
          prefetch_l1(p.u[d] + idx[0]);
          prefetch_l1(p.u[d] + idx[1]);
        }
        {
          float2 o[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) o[d] = make_float2(p.o[d][idx[0]], p.o[d][idx[1]]);
          int r[3] = {l[0], l[1], l[2]};
          // axes 0, 1, 2 of the arrays: d, e, f; the weights are formed again for
          // every rotation and component (kept, they would cost the third CTA)
#pragma unroll 1
          for (int d = 0; d < 3; ++d) {
            const int sd = L.sd(d, 4), se = L.se(d, 4);
            // node-centred axes start at c-1, half-staggered ones at c-2
            const float* b = sF + L.start(d, 4) + r[0] * sd + r[1] * se + r[2];
            E[0] = E[1], E[1] = E[2];
            B[0] = B[1], B[1] = B[2];
            {
              float2 wd[5], we[4], wf[4];
              half_weights32(o[0], wd);
              spline32(o[1], we);
              spline32(o[2], wf);
              E[2] = gather_pair<5, 4, 4>(b + se + 1, sd, se, wd, we, wf);
            }
            {
              float2 wd[4], we[5], wf[5];
              spline32(o[0], wd);
              half_weights32(o[1], we);
              half_weights32(o[2], wf);
              B[2] = gather_pair<4, 5, 5>(b + L.part(d, 4) + sd, sd, se, wd, we, wf);
            }
            const int r0 = r[0];
            r[0] = r[1], r[1] = r[2], r[2] = r0;
            const float2 t = o[0];
            o[0] = o[1], o[1] = o[2], o[2] = t;
          }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d] = make_float2(p.u[d][idx[0]], p.u[d][idx[1]]);
        const float2 ig = boris32(pc.h, E, B, u);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (k == 1 && !have[1]) break;
          const float igk = k ? ig.y : ig.x;
          if (igk > 0.0f) {
            const float uk[3] = {k ? u[0].y : u[0].x, k ? u[1].y : u[1].x, k ? u[2].y : u[2].x};
            key[k] = finish(l, idx[k], pos[k], ent[k], uk, igk, true);
          } else {  // not finite: once more, alone
            order[pos[k]] = ent[k] | kCross | kSteps;
            sc[7] = 1;
          }
          if (key[k] == t) own += 1;
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) count_leaving(cnt_next, key[k], t);
    }
    __syncthreads();
    // A pair's windows also read nodes at weight zero, where a NaN or an infinity is
    // none of the particle's business: those whose momentum came out not finite are
    // pushed with their own windows.  What stays so is reported, and absorbed without
    // moving or depositing.  (Here, and not where it was found: a branch there costs the
    // others 3 %.)
    if (sc[7]) {
      for (int pos = tid; pos < nch; pos += kPushThreads) {
        if ((order[pos] & (kCross | kStray | kSteps)) != (kCross | kSteps)) continue;
        const unsigned ent = order[pos] & ~(kCross | kSteps);
        const int idx = c0 + (int)(ent & 4095);
        order[pos] = ent;
        int l[3];
        L.cell((ent >> 12) & 4095, l);
        float2 o[3], u2[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) o[d] = dup2(p.o[d][idx]), u2[d] = dup2(p.u[d][idx]);
        const float ig = push_own32(sF, L, l, pc.h, o, u2);
        const bool good = ig > 0.0f;
        if (!good) atomicOr(err, 8);
        const float u[3] = {good ? u2[0].x : 0.0f, good ? u2[1].x : 0.0f, good ? u2[2].x : 0.0f};
        const int key = finish(l, idx, pos, ent, u, ig, good);
        if (key >= 0) atomicAdd(cnt_next + key, 1);
      }
      __syncthreads();
    }
    if (npass > 1) {
      keep_lists(P, p, c0, nch, nitem, pairB);
      __syncthreads();
    }
  }

  // ---- the region becomes the J tile ----
  {
    int4* z = reinterpret_cast<int4*>(smem_raw);
    const int n = (int)(so.order / 16);
    for (int i = tid; i < n; i += kPushThreads) z[i] = make_int4(0, 0, 0, 0);
  }
  for (int ps = 0; ps < npass; ++ps) {
    const Pass pass(ps, npass, ntile);
    const int nch = pass.n, c0 = pbeg + pass.begin;
    if (npass > 1) {
      __syncthreads();
      fetch_lists(P, p, c0, nch, pairB);
    }
    __syncthreads();
    const int ranked = sc[33];
    const int nround = sc[16 + kRanks / 2];
    const int nitem = nround + (nch - ranked);
    const float third = 1.0f / 3.0f;
    int round = 0;
    for (int i = tid; i < nitem; i += kPushThreads) {
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
      const bool dep[2] = {!(ent[0] & kCross), pb != 0xffff && !(ent[1] & kCross)};
      if (!(dep[0] || dep[1])) continue;
      int r[3];
      L.cell((ent[0] >> 12) & 4095, r);
      float2 oa[3], ob[3], qw;  // old and new offsets
      {
        const int i0 = c0 + (int)(ent[0] & 4095), i1 = c0 + (int)(ent[1] & 4095), d0 = c0 + pos[0], d1 = c0 + pos[1];
        qw = make_float2(dep[0] ? pc.q * p.w[i0] : 0.0f, dep[1] ? pc.q * p.w[i1] : 0.0f);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          oa[d] = make_float2(p.o[d][i0], p.o[d][i1]);
          ob[d] = make_float2(dep[0] ? pn.o[d][d0] : oa[d].x, dep[1] ? pn.o[d][d1] : oa[d].y);
        }
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {  // axes 0, 1, 2 of the arrays: d, e, f
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + (r[0] + 1) * sd + (r[1] + 1) * se + r[2] + 1;  // nodes c-1 .. c+2
        const int sh = sc[50 + d] + 31 - sc[4 + d];
        const long long half = (long long)(1u << (sh - 1));
        int Pi[2][3];
        {
          float2 S[4], D[4];
          shapes32(oa[0], ob[0], S, D);
          const float scale = __int_as_float((127 + sc[50 + d]) << 23);
          const float jc = d == 0 ? pc.jc[0] : (d == 1 ? pc.jc[1] : pc.jc[2]);
          const float2 c = mul2(mul2(dup2(jc), qw), dup2(scale));
          float2 run = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            run = add2(run, D[m]);
            const float2 v = mul2(c, run);
            Pi[0][m] = __float2int_rn(v.x);
            Pi[1][m] = __float2int_rn(v.y);
          }
        }
        // A(b, c) = S_e (S_f + D_f / 2) + D_e (S_f / 2 + D_f / 3)
        float2 ak[4], bk[4];
        {
          float2 S[4], D[4];
          shapes32(oa[2], ob[2], S, D);
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            ak[m] = mul2(dup2(kA31), fma2(dup2(0.5f), D[m], S[m]));
            bk[m] = mul2(dup2(kA31), fma2(dup2(third), D[m], mul2(dup2(0.5f), S[m])));
          }
        }
        float2 S[4], D[4];
        shapes32(oa[1], ob[1], S, D);
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float2 A = fma2(D[b], bk[c], mul2(S[b], ak[c]));
            const int A0 = __float2int_rn(A.x), A1 = __float2int_rn(A.y);
#pragma unroll
            for (int m = 0; m < 3; ++m)
              add_current(j + m * sd + b * se + c, lo, mad_wide(Pi[1][m], A1, mad_wide(Pi[0][m], A0, half)), sh);
          }
        const int r0 = r[0];
        r[0] = r[1], r[1] = r[2], r[2] = r0;
        const float2 t = oa[0], v = ob[0];
        oa[0] = oa[1], oa[1] = oa[2], oa[2] = t;
        ob[0] = ob[1], ob[1] = ob[2], ob[2] = v;
      }
    }
    // particles that left their cell, on 5-node windows where they moved, and light ones
    const int ncross = sc[1];
    for (int i = tid; i < ncross; i += kPushThreads) {
      const int pos = P.cross[i];
      const unsigned e = order[pos];
      int r[3], n[3];
      L.cell((e >> 12) & 4095, r);
      const int idx = c0 + (int)(e & 4095), dst = c0 + pos;
      const float qw = pc.q * p.w[idx];
      float S[3][5], D[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int dc = (int)((e >> (24 + 2 * d)) & 3u) - 1;
        float2 w[4];  // at the old and the new offset
        spline32(make_float2(p.o[d][idx], pn.o[d][dst]), w);
        const int p0 = dc < 0 ? 1 : 0, p1 = dc > 0 ? 1 : 0;
        r[d] += 1 - p0;
        n[d] = dc != 0 ? 5 : 4;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const float a0 = p0 ? (m > 0 ? w[m > 0 ? m - 1 : 0].x : 0.0f) : (m < 4 ? w[m < 4 ? m : 3].x : 0.0f);
          const float a1 = p1 ? (m > 0 ? w[m > 0 ? m - 1 : 0].y : 0.0f) : (m < 4 ? w[m < 4 ? m : 3].y : 0.0f);
          S[d][m] = a0;
          D[d][m] = a1 - a0;
        }
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + r[0] * sd + r[1] * se + r[2];
        int Pi[4], sh;
        {
          const float jq = (d == 0 ? pc.jc[0] : (d == 1 ? pc.jc[1] : pc.jc[2])) * qw;
          const int ep = ((__float_as_int(0.76f * jq) >> 23) & 255) - 127, s = sc[4 + d];
          const int kp = max(min(30 - ep, s), sc[50 + d]);
          sh = kp + 31 - s;
          const float c = jq * __int_as_float((127 + kp) << 23);
          float run = 0.0f;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            run += D[0][m];
            Pi[m] = __float2int_rn(c * run);
          }
        }
        float ak[5], bk[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          ak[m] = kA31 * (S[2][m] + 0.5f * D[2][m]);
          bk[m] = kA31 * (0.5f * S[2][m] + third * D[2][m]);
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
                  if (m < n[0] - 1)
                    add_current(j + m * sd + b * se + c, lo, mad_wide(Pi[m], A, (long long)(1u << (sh - 1))), sh);
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
  }
  __syncthreads();

  // flush: a half warp per (x, y) row, the lanes along z
  {
    const int NX = tl.tx + 5, NZ = tl.tz + 5;
    for (RowWalk r(tl.ty + 5); r.lx < NX; r.next()) {
      const int lx = r.lx, ly = r.ly;
      const int gi0 = P.tabx[lx] + P.taby[ly];
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
            atomicAdd(f.c[JX + d] + gi0 + P.tabz[lz], v * __int_as_float((127 - sc[4 + d]) << 23));  // 2^-s
          }
        }
      }
    }
  }
  own = __reduce_add_sync(0xffffffffu, own);
  if (lane == 0 && own) atomicAdd(cnt_next + t, own);
}

}  // namespace pic
