// pic_push64.cuh -- the FP64 particle push: gather, Boris push, move and
// Esirkepov deposit of one cell tile per CTA, with the gather and the deposit
// in 64-bit fixed point on the integer pipes (pic_fixed64.cuh).
//
// The staged E and B become int64 at a power of two 2^sF per tile and
// component with max|F| 2^sF < 2^60, and the J tile holds exact 64-bit sums as
// three 32-bit words at 2^s per tile and component with B 2^s < 2^62, B a bound on
// every node's sum taken from the particles' speeds before the push: a cold or
// slow tile gets a fine scale, not one sized for moves of a whole cell.
//
// What bounded the one-pass kernel that this replaces: instructions, about
// 20,000 per particle, issued 36 % of the time (16 warps per SM, waits for
// instructions and for the shared-memory adds' returns).  What changed:
// - one instruction per 32x32->64 product (mad_wide: from the plain expression
//   the compiler made 16 of 3) and centred splits at 32 bits, whose products
//   need no 64-bit shifts;
// - the weights of two axes are multiplied once for the two components that
//   share them (E_d and B_e), and the gather then sums 16 products per node of
//   the third axis: 48 products of weights and 408 of values, from 504;
// - the shape factors are formed in fixed point: 90 FP64 instructions per
//   particle, from 230;
// - particles that stay in their cell (4-node windows) deposit apart from those
//   that leave it (5-node windows), which made every warp run the wide loops;
// - a current word pair with a carry became three overlapping words added by
//   reductions that return nothing.
//
// Measured (the push of a step, the one-pass kernel -> this one): 119 M particles,
// 1536x256x256 cells 167 -> 69 ms; whole steps, with the field update's change: 118 M
// 183 -> 78.6 ms, 7 M, 384x96x96 10.6 -> 4.8 ms, 436 k at random places 0.97 -> 0.54 ms.
// In a run's state 9,380 instructions per 32 particles, issued 40 % of the time; the
// shared-memory pipe is 54 % busy, no other above a third (integer ALU 31 %, FMA 27 %,
// FP64 26 %): fixed latencies at 16 warps per SM bound it.
#pragma once

#include "pic_push.cuh"

namespace pic {

constexpr int kJ64Range = 62;  // J sums

// Scale exponent of the J tile for component c: B 2^s < 2^62 with B = 1.001 |q|
// S / (dt d_b d_c), S a bound on sum |w| |running sum|.  A particle moves at
// most dt/d |u'| cells along an axis, |u'| <= |u| + 2 |h| |E| (the Boris
// rotation keeps |u|), and a running sum of the deposit changes by at most 3/4
// of the move (the slope bound of the cubic spline's partial sums); 2^-20
// covers the rounding.  su = sum |w| min(1, |u|), sw = sum |w|, kick >= 2 |h| |E|.
__device__ __forceinline__ int j64_scale(const PushCoef<double>& pc, int c, float su, float sw, float kick) {
  const float dtd = (float)(c == 0 ? pc.dtd[0] : (c == 1 ? pc.dtd[1] : pc.dtd[2]));
  const float S = 0.75f * (dtd * fminf(su + kick * sw, sw) + 0x1p-20f * sw);
  const float B = 1.001f * fabsf((float)pc.q) * S * fabsf((float)(c == 0 ? pc.jc[0] : (c == 1 ? pc.jc[1] : pc.jc[2])));
  const int eb = ((__float_as_int(B) >> 23) & 255) - 127;  // B in [2^eb, 2^(eb+1))
  return B > 0.0f ? kJ64Range - 1 - eb : 0;
}

// Exact 64-bit add of X as three overlapping words, X mod 2^32, X >> 20 and
// X >> 40 mod 2^32, by reductions that return nothing (an add of two words
// waits for the low word's old value to form the carry).
__device__ __forceinline__ void add_current64(unsigned* j, int part, long long X) {
  const unsigned l = (unsigned)X, h = (unsigned)((unsigned long long)X >> 32);
  red_u32(j, l);
  red_u32(j + part, __funnelshift_r(l, h, 20));
  red_u32(j + 2 * part, (unsigned)((int)h >> 8));
}

// The sum of X from the words' sums of up to kChunk + 1 adds: sum (X >> 40) is exact
// (the sum itself is below 2^62); sum (X >> 20) lies within n 2^20 < 2^32 above
// 2^20 times it, and sum X within n 2^20 above 2^20 times that.
__device__ __forceinline__ long long sum_current64(unsigned w0, unsigned w1, unsigned w2) {
  const long long a = (long long)(int)w2 << 20;
  const long long b = a + (long long)(w1 - (unsigned)a);
  const long long c = b << 20;
  return c + (long long)(w0 - (unsigned)c);
}
static_assert(kChunk + 1 < 4096, "the words' overlap holds the carries of 2^12 adds");

template <bool FIXED>
__global__ void __launch_bounds__(kPushThreads, 2)
    k_push64(Geom<double> g, Tiles tl, Fields<double> f, Parts<double> p, Parts<double> pn,
             const int* __restrict__ tstart, int capacity, int* __restrict__ keys, int* __restrict__ cnt_next,
             PushCoef<double> pc, int origin_after, int xlo, int xhi, unsigned long long* pushed, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (g.dyn) origin_after = g.dyn->origin_after;
  const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int pbeg = min(tstart[t], capacity), pend = min(tstart[t + 1], capacity);
  if (pbeg >= pend) return;
  const PushLayout<double, FIXED> L(tl);
  const PushTile P = push_tile<double, FIXED>(smem_raw, g, tl, t);
  const PushSmem so = PushSmem::of<double, FIXED>(tl);
  long long* sF = reinterpret_cast<long long*>(smem_raw);
  unsigned* sJ = reinterpret_cast<unsigned*>(smem_raw);
  unsigned* order = P.order;
  int* sc = P.sc;
  const int W = L.words();
  const int ntile = pend - pbeg;
  if (tid == 0) atomicAdd(pushed, (unsigned long long)ntile);
  const int npass = (ntile + kChunk - 1) / kChunk;
  int own = 0;

  for (int ps = 0; ps < npass; ++ps) {
    const Pass pass(ps, npass, ntile);
    const int nch = pass.n, c0 = pbeg + pass.begin;
    rank_clear(P, W);
    __syncthreads();

    // Stage E_d (part 0) and B_e, e the axis after d (part 1): a half warp per
    // (x, y) row, the lanes along z; take the largest exponent of each.
    const int SX = tl.tx + 4, SZ = tl.tz + 4;
    if (ps == 0) {
      int emax[6] = {0, 0, 0, 0, 0, 0};
      for (RowWalk r(tl.ty + 4); r.lx < SX; r.next()) {
        const int lx = r.lx, ly = r.ly;
        const int gi0 = P.tabx[lx] + P.taby[ly];
        for (int lz = tid & 15; lz < SZ; lz += 16) {
          const int gi = gi0 + P.tabz[lz];
          const int i3[3] = {lx, ly, lz};
          long long v[6];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            v[2 * d] = __double_as_longlong(f.c[EX + d][gi]);
            v[2 * d + 1] = __double_as_longlong(f.c[BX + (d + 1) % 3][gi]);
          }
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const int d = k >> 1;
            sF[L.start(d, 4) + (k & 1) * L.part(d, 4) + i3[d] * L.sd(d, 4) + i3[(d + 1) % 3] * L.se(d, 4) +
               i3[(d + 2) % 3]] = v[k];
            emax[k] = max(emax[k], (int)((unsigned long long)v[k] >> 52) & 0x7FF);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const unsigned e = __reduce_max_sync(0xffffffffu, (unsigned)emax[k]);
        if (lane == 0) atomicMax(sc + 50 + k, (int)e);
      }
    }
    int sr[kPerThread];
    rank_count(P, L, g, tl, p.cell, c0, nch, sr, err);
    if (ps == 0) {  // over the tile
      float su = 0.0f, sw = 0.0f;
      for (int k = tid; k < ntile; k += kPushThreads) {
        const float wa = fabsf((float)p.w[pbeg + k]);
        const float ux = (float)p.u[0][pbeg + k], uy = (float)p.u[1][pbeg + k], uz = (float)p.u[2][pbeg + k];
        su += wa * fminf(1.0f, sqrtf(ux * ux + uy * uy + uz * uz));
        sw += wa;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        su += __shfl_down_sync(0xffffffffu, su, o);
        sw += __shfl_down_sync(0xffffffffu, sw, o);
      }
      if (lane == 0) {
        atomicAdd(reinterpret_cast<float*>(sc + 2), su);
        atomicAdd(reinterpret_cast<float*>(sc + 3), sw);
      }
    }
    __syncthreads();
    rank_masks(P, W);
    if (ps == 0 && tid < 3) {
      // |E| <= sqrt 3 max_c |E_c| < sqrt 3 2^(emax - 1022)
      const int eE = max(max(sc[50], sc[52]), sc[54]);
      const float kick = eE == 0 ? 0.0f : ldexpf(3.4642f * fabsf((float)pc.h), eE - 1022);
      sc[4 + tid] = j64_scale(pc, tid, __int_as_float(sc[2]), __int_as_float(sc[3]), kick);
    }
    if (ps == 0 && tid < 6) {
      // max|F| 2^sF < 2^60; a non-finite value is reported
      const int e = sc[50 + tid];
      if (e == 0x7FF) atomicOr(err, 8);
      sc[56 + tid] = kFieldBits - 1 - (max(e, kFieldMinExp) - 1023);
    }
    __syncthreads();
    rank_order(P, W, nch, sr);
    if (ps == 0) {
      // the staged doubles become split fixed-point words in place
      int emax[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) emax[k] = max(sc[50 + k], kFieldMinExp);
      for (RowWalk r(tl.ty + 4); r.lx < SX; r.next()) {
        const int lx = r.lx, ly = r.ly;
        for (int lz = tid & 15; lz < SZ; lz += 16) {
          const int i3[3] = {lx, ly, lz};
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const int d = k >> 1;
            long long* w = sF + L.start(d, 4) + (k & 1) * L.part(d, 4) + i3[d] * L.sd(d, 4) +
                           i3[(d + 1) % 3] * L.se(d, 4) + i3[(d + 2) % 3];
            const S32 x = split32(field_fixed(*w, emax[k]));
            *reinterpret_cast<int2*>(w) = make_int2(x.lo, x.hi);
          }
        }
      }
    }
    __syncthreads();

    // ---- gather, push, move ----
    for (int i0 = 0; i0 < nch; i0 += kPushThreads) {
      const int pos = i0 + tid;
      bool have = pos < nch;
      const unsigned ent = have ? order[pos] : kStray;
      if (have && (ent & kStray)) {  // dropped with the error bit set
        keys[c0 + pos] = -1;
        order[pos] = ent | kCross;
      }
      have = have && !(ent & kStray);
      int key = -2;
      if (have) {
        int l[3];
        L.cell((ent >> 12) & 4095, l);
        const int idx = c0 + (int)(ent & 4095), dst = c0 + pos;
        double E[3], B[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) prefetch_l1(p.u[d] + idx);  // for after the gather
        {
          long long T[3];  // offsets at 2^63
          int r[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            T[d] = offset63(p.o[d][idx]);
            r[d] = l[d];
          }
          // Axes 0, 1, 2 of the arrays: d, e, f.  E_d sits on half nodes of d and
          // nodes of e, f; B_e on half nodes of d and f and nodes of e: the two
          // share the weights of (d, e).  The weights are formed again for every
          // rotation: kept, they would fill the registers.
#pragma unroll 1
          for (int d = 0; d < 3; ++d) {
            const int sd = L.sd(d, 4), se = L.se(d, 4);
            // half nodes see the offset t + 1/2 from c-2 (t < 1/2) or t - 1/2 from c-1: u = t or t - 1
            const bool low0 = T[0] < kHalf63, low2 = T[2] < kHalf63;
            const int2* b = reinterpret_cast<const int2*>(sF) + L.start(d, 4) + (r[0] + (low0 ? 0 : 1)) * sd +
                            (r[1] + 1) * se + r[2];
            S32 wde[4][4], wf[4];
            {
              S32 wd[4], we[4];
              spline63(low0 ? T[0] : T[0] - kHalf63 - kHalf63, wd);
              spline63(T[1] - kHalf63, we);
#pragma unroll
              for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) wde[i][j] = split32(2 * floor64(wd[i], we[j]));
            }
            spline63(T[2] - kHalf63, wf);
            const double e = fixed_to_double(gather64(b + 1, sd, se, wde, wf), sc[56 + 2 * d]);
            spline63(low2 ? T[2] : T[2] - kHalf63 - kHalf63, wf);
            const double m =
                fixed_to_double(gather64(b + L.part(d, 4) + (low2 ? 0 : 1), sd, se, wde, wf), sc[57 + 2 * d]);
            E[0] = E[1], E[1] = E[2], E[2] = e;
            B[1] = B[2], B[2] = B[0], B[0] = m;  // B_y, B_z, B_x come in this order
            const int r0 = r[0];
            r[0] = r[1], r[1] = r[2], r[2] = r0;
            const long long t0 = T[0];
            T[0] = T[1], T[1] = T[2], T[2] = t0;
          }
        }
        double u[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d] = p.u[d][idx];
        // relativistic Boris push
        const double h = pc.h;
        double um[3], tv[3], sv[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) um[d] = u[d] + h * E[d];
        const double hg = h * rsqrt(1.0 + um[0] * um[0] + um[1] * um[1] + um[2] * um[2]);  // h / gamma-
#pragma unroll
        for (int d = 0; d < 3; ++d) tv[d] = hg * B[d];
        const double s2 = 2.0 / (1.0 + tv[0] * tv[0] + tv[1] * tv[1] + tv[2] * tv[2]);
#pragma unroll
        for (int d = 0; d < 3; ++d) sv[d] = s2 * tv[d];
        const double px = um[0] + (um[1] * tv[2] - um[2] * tv[1]);
        const double py = um[1] + (um[2] * tv[0] - um[0] * tv[2]);
        const double pz = um[2] + (um[0] * tv[1] - um[1] * tv[0]);
        u[0] = um[0] + (py * sv[2] - pz * sv[1]) + h * E[0];
        u[1] = um[1] + (pz * sv[0] - px * sv[2]) + h * E[1];
        u[2] = um[2] + (px * sv[1] - py * sv[0]) + h * E[2];
        double ig = rsqrt(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);  // 1 / gamma
        const bool good = ig > 0.0;
        if (!good) {  // a non-finite momentum: reported; absorbed without moving or depositing
          atomicOr(err, 8);
          ig = 0.0;
          u[0] = u[1] = u[2] = 0.0;
        }
        int dc[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {  // |move| < 1 cell per axis
          double o = p.o[d][idx] + pc.dtd[d] * u[d] * ig;
          int k = 0;
          if (lt_zero(o)) {
            o += 1.0;
            k = -1;
          } else if (ge_one(o)) {
            o -= 1.0;
            k = 1;
          }
          if (ge_one(o)) {
            o = 0.0;
            k += 1;
          }
          dc[d] = k;
          pn.o[d][dst] = o;
          pn.u[d][dst] = u[d];
        }
        pn.w[dst] = p.w[idx];
        if (pn.id) pn.id[dst] = p.id[idx];
        key = place_moved(P, g, tl, t, l, dc, good, false, origin_after, xlo, xhi, pos, ent, pn.cell + dst, keys + dst);
        if (key == t) own += 1;
      }
      count_leaving(cnt_next, key, t);
    }
    __syncthreads();
    if (npass > 1) {
      keep_lists(P, p, c0, nch, 0, nullptr);
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
      if (ps > 0) {  // the sums so far as the words of one add (see sum_current64)
#pragma unroll 1
        for (int d = 0; d < 3; ++d) {
          const int n = L.part(d, 5);
          unsigned* w = sJ + L.start(d, 5);
          for (int i = tid; i < n; i += kPushThreads) {
            const long long X = sum_current64(w[i], w[i + n], w[i + 2 * n]);
            w[i] = (unsigned)X;
            w[i + n] = (unsigned)(X >> 20);
            w[i + 2 * n] = (unsigned)(X >> 40);
          }
        }
      }
      fetch_lists(P, p, c0, nch, (unsigned short*)nullptr);
    }
    __syncthreads();
    // 2 P 2^s = 2 q w jc run 2^s, below 2^63 by the choice of the scale; run at 2^62
    for (int pos = tid; pos < nch; pos += kPushThreads) {
      const unsigned ent = order[pos];
      if (pos + kPushThreads < nch) {  // the next particle's records
        const int ni = c0 + (int)(order[pos + kPushThreads] & 4095);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          prefetch_l1(p.o[d] + ni);
          prefetch_l1(pn.o[d] + c0 + pos + kPushThreads);
        }
        prefetch_l1(p.w + ni);
      }
      if (ent & kCross) continue;
      int r[3];
      L.cell((ent >> 12) & 4095, r);
      const int idx = c0 + (int)(ent & 4095), dst = c0 + pos;
      const double qw = pc.q * p.w[idx];
      long long S[3][4], D[3][4];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        long long w1[4];
        spline_fixed<62>(offset63(p.o[d][idx]) - kHalf63, S[d]);
        spline_fixed<62>(offset63(pn.o[d][dst]) - kHalf63, w1);
#pragma unroll
        for (int k = 0; k < 4; ++k) D[d][k] = w1[k] - S[d][k];
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {  // axes 0, 1, 2 of the arrays: d, e, f
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + (r[0] + 1) * sd + (r[1] + 1) * se + r[2] + 1;  // nodes c-1 .. c+2
        S32 Pi[3];
        {
          const double cfs = qw * ((d == 0 ? pc.jc[0] : (d == 1 ? pc.jc[1] : pc.jc[2])) * exp2i(sc[4 + d] - 61));
          long long run = 0;
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            run += D[0][m];
            Pi[m] = split32(to_fixed(fixed_to_double(run, 0) * cfs, 0));
          }
        }
        S32 ak[4], bk[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          // at 2^63: S_f + D_f / 2 and S_f / 2 + D_f / 3 (= S1 - D / 3 at 2^62)
          const long long S1 = S[2][c] + D[2][c];
          ak[c] = split32(S[2][c] + S1);
          bk[c] = split32(S1 - floor64(split32(D[2][c]), third64()));
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const S32 sb = split32(S[1][b]), db = split32(D[1][b]);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            Acc32 a = {0LL, 0LL};
            acc32(a, sb, ak[c]);
            acc32(a, db, bk[c]);
            const S32 A = split32(acc32_result(a) << 2);  // at 2^63
#pragma unroll
            for (int m = 0; m < 3; ++m) add_current64(j + m * sd + b * se + c, lo, mul64(Pi[m], A));
          }
        }
        const int r0 = r[0];
        r[0] = r[1], r[1] = r[2], r[2] = r0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const long long v = S[0][k], w = D[0][k];
          S[0][k] = S[1][k], S[1][k] = S[2][k], S[2][k] = v;
          D[0][k] = D[1][k], D[1][k] = D[2][k], D[2][k] = w;
        }
      }
    }
    // particles that left their cell: 5-node windows where they moved
    const int ncross = sc[1];
    for (int i = tid; i < ncross; i += kPushThreads) {
      const int pos = P.cross[i];
      const unsigned ent = order[pos];
      int r[3], n[3];
      L.cell((ent >> 12) & 4095, r);
      const int idx = c0 + (int)(ent & 4095), dst = c0 + pos;
      const double qw = pc.q * p.w[idx];
      long long S[3][5], D[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int dc = (int)((ent >> (24 + 2 * d)) & 3u) - 1;
        long long w0[4], w1[4];
        spline_fixed<62>(offset63(p.o[d][idx]) - kHalf63, w0);
        spline_fixed<62>(offset63(pn.o[d][dst]) - kHalf63, w1);
        const int p0 = dc < 0 ? 1 : 0, p1 = dc > 0 ? 1 : 0;
        r[d] += 1 - p0;
        n[d] = dc != 0 ? 5 : 4;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const long long a0 = p0 ? (m > 0 ? w0[m > 0 ? m - 1 : 0] : 0LL) : (m < 4 ? w0[m < 4 ? m : 3] : 0LL);
          const long long a1 = p1 ? (m > 0 ? w1[m > 0 ? m - 1 : 0] : 0LL) : (m < 4 ? w1[m < 4 ? m : 3] : 0LL);
          S[d][m] = a0;
          D[d][m] = a1 - a0;
        }
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + r[0] * sd + r[1] * se + r[2];
        S32 Pi[4];
        {
          const double cfs = qw * ((d == 0 ? pc.jc[0] : (d == 1 ? pc.jc[1] : pc.jc[2])) * exp2i(sc[4 + d] - 61));
          long long run = 0;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            run += D[0][m];
            Pi[m] = split32(to_fixed(fixed_to_double(run, 0) * cfs, 0));
          }
        }
        S32 ak[5], bk[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const long long S1 = S[2][c] + D[2][c];
          ak[c] = split32(S[2][c] + S1);
          bk[c] = split32(S1 - floor64(split32(D[2][c]), third64()));
        }
#pragma unroll
        for (int b = 0; b < 5; ++b)
          if (b < n[1]) {
            const S32 sb = split32(S[1][b]), db = split32(D[1][b]);
#pragma unroll
            for (int c = 0; c < 5; ++c)
              if (c < n[2]) {
                Acc32 a = {0LL, 0LL};
                acc32(a, sb, ak[c]);
                acc32(a, db, bk[c]);
                const S32 A = split32(acc32_result(a) << 2);
#pragma unroll
                for (int m = 0; m < 4; ++m)
                  if (m < n[0] - 1) add_current64(j + m * sd + b * se + c, lo, mul64(Pi[m], A));
              }
          }
        const int r0 = r[0], n0 = n[0];
        r[0] = r[1], r[1] = r[2], r[2] = r0;
        n[0] = n[1], n[1] = n[2], n[2] = n0;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const long long v = S[0][k], w = D[0][k];
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
          const long long X = sum_current64(w[0], w[L.part(d, 5)], w[2 * L.part(d, 5)]);
          if (X != 0) atomicAdd(f.c[JX + d] + gi0 + P.tabz[lz], fixed_to_double(X, sc[4 + d]));
        }
      }
    }
  }
  own = __reduce_add_sync(0xffffffffu, own);
  if (lane == 0 && own) atomicAdd(cnt_next + t, own);
}

}  // namespace pic
