// pic_push64.cuh -- the FP64 particle push: gather, Boris push, move and
// Esirkepov deposit of one cell tile per CTA, with the gather and the deposit
// in 64-bit fixed point on the integer pipes (pic_fixed64.cuh).
//
// The staged E and B become int64 at a power of two 2^sF per tile and
// component with max|F| 2^sF < 2^58, and the J tile holds exact 64-bit sums as
// two 32-bit words at 2^s per pass and component with B 2^s < 2^62, B a bound on
// every node's sum taken from the particles' speeds before the push: a cold or
// slow tile gets a fine scale, not one sized for moves of a whole cell.
//
// What bounded the one-pass kernel that this replaces: instructions, about
// 20,000 per particle, issued 36 % of the time (16 warps per SM, waits for
// instructions and for the shared-memory adds' returns).  What changed:
// - one 32x32->64 multiply-add per product, spelt out (mad_wide), and values
//   split at 31 bits, so that the two cross products share an accumulator;
// - the weights of two axes are multiplied once for the two components that
//   share them (E_d and B_e), and the gather then sums 16 products per node of
//   the third axis: 96 products of weights and 408 of values, from 504;
// - the shape factors are formed in fixed point: 130 FP64 instructions per
//   particle, from 230;
// - particles that stay in their cell (4-node windows) deposit apart from those
//   that leave it (5-node windows), which made every warp run the wide loops;
// - the lanes of a warp hold neighbouring cells, and the returns of a node
//   column's adds are waited for together.
//
// Measured (whole step, before -> after): 118 M particles, 1536x256x256 cells
// 183 -> 113 ms; 7 M, 384x96x96 10.6 -> 6.4 ms; 126 k, 128x32x32 0.368 ->
// 0.251 ms.  Issue is active 42 % of cycles, the integer ALU 43 %, the FP64 pipe
// 25 %; the top stalls are fixed latencies and the adds' returns.
#pragma once

#include "pic_push.cuh"

namespace pic {

constexpr int kField64Range = 58;  // staged fields: 16-term sums need |x| < 2^58
constexpr int kJ64Range = 62;      // J sums of single products

// Scale exponent of the J tile for component c: B 2^s < 2^62 with B = 1.001 |q|
// S / (dt d_b d_c), S a bound on sum |w| |running sum|.  A particle moves at
// most dt/d |u'| cells along an axis, |u'| <= |u| + 2 |h| |E| (the Boris
// rotation keeps |u|), and a running sum of the deposit changes by at most 3/4
// of the move (the slope bound of the cubic spline's partial sums); 2^-20
// covers the rounding.  su = sum |w| min(1, |u|), sw = sum |w|, kick >= 2 |h| |E|.
__device__ __forceinline__ int j64_scale(const Geom<double>& g, double q, int c, float su, float sw, float kick) {
  const float dtd = (float)(g.dt / (c == 0 ? g.dx : (c == 1 ? g.dy : g.dz)));
  const float S = 0.75f * (dtd * fminf(su + kick * sw, sw) + 0x1p-20f * sw);
  const double jcc = c == 0 ? g.dt * g.dy * g.dz : (c == 1 ? g.dt * g.dx * g.dz : g.dt * g.dx * g.dy);
  const float B = 1.001f * fabsf((float)q) * S / (float)jcc;
  const int eb = ((__float_as_int(B) >> 23) & 255) - 127;  // B in [2^eb, 2^(eb+1))
  return B > 0.0f ? kJ64Range - 1 - eb : 0;
}

// Exact 64-bit adds of X[0 .. N) into the shared word pairs at lo + m stride
// (hi words hi_off further): the low words' adds return the old values, which
// give the carries; the N returns are waited for together.
template <int N>
__device__ __forceinline__ void add_current64(unsigned* hi, int lo_off, int stride, const long long (&X)[N], int n) {
  unsigned old[N];
#pragma unroll
  for (int m = 0; m < N; ++m)
    if (m < n) old[m] = atom_add_u32_shared(hi + lo_off + m * stride, (unsigned)X[m]);
#pragma unroll
  for (int m = 0; m < N; ++m)
    if (m < n) {
      const unsigned l = (unsigned)X[m], h = (unsigned)((unsigned long long)X[m] >> 32);
      red_add_u32_shared(hi + m * stride, h + (old[m] + l < l ? 1u : 0u));
    }
}

template <bool FIXED>
__global__ void __launch_bounds__(kPushThreads, 2)
    k_push64(Geom<double> g, Tiles tl, Fields<double> f, Parts<double> p, Parts<double> pn,
             const int* __restrict__ tstart, int capacity, int* __restrict__ keys, int* __restrict__ cnt_next,
             double h, double q, int origin_after, int xlo, int xhi, unsigned long long* pushed, int* err) {
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
  const int npass = (ntile + kChunk - 1) / kChunk, per_pass = (ntile + npass - 1) / npass;
  int own = 0;

  for (int ch0 = 0; ch0 < ntile; ch0 += per_pass) {
    const int nch = min(per_pass, ntile - ch0), c0 = pbeg + ch0;
    rank_clear(P, W);
    __syncthreads();

    // Stage E_d (part 0) and B_e, e the axis after d (part 1): a half warp per
    // (x, y) row, the lanes along z; take the largest exponent of each.
    const int SY = tl.ty + 4, rows = (tl.tx + 4) * SY, SZ = tl.tz + 4;
    {
      int emax[6] = {0, 0, 0, 0, 0, 0};
      for (int r = tid >> 4; r < rows; r += kPushThreads / 16) {
        const int lx = r / SY, ly = r - lx * SY;
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
    {
      float su = 0.0f, sw = 0.0f;
      for (int k = tid; k < nch; k += kPushThreads) {
        const float wa = fabsf((float)p.w[c0 + k]);
        const float ux = (float)p.u[0][c0 + k], uy = (float)p.u[1][c0 + k], uz = (float)p.u[2][c0 + k];
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
    if (tid < 3) {
      // |E| <= sqrt 3 max_c |E_c| < sqrt 3 2^(emax - 1022)
      const int eE = max(max(sc[50], sc[52]), sc[54]);
      const float kick = eE == 0 ? 0.0f : ldexpf(3.4642f * fabsf((float)h), eE - 1022);
      sc[4 + tid] = j64_scale(g, q, tid, __int_as_float(sc[2]), __int_as_float(sc[3]), kick);
    }
    if (tid < 6) {
      // max|F| 2^sF < 2^58; an all-zero component takes sF = 1000; a non-finite value is reported
      const int e = sc[50 + tid];
      if (e == 0x7FF) atomicOr(err, 8);
      sc[56 + tid] = e == 0 ? 1000 : min(kField64Range - 1 - (e - 1023), 1000);
    }
    __syncthreads();
    rank_order(P, W, nch, sr);
    {
      // the staged doubles become split fixed-point words in place
      int k58[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) k58[k] = sc[56 + k];
      for (int r = tid >> 4; r < rows; r += kPushThreads / 16) {
        const int lx = r / SY, ly = r - lx * SY;
        for (int lz = tid & 15; lz < SZ; lz += 16) {
          const int i3[3] = {lx, ly, lz};
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const int d = k >> 1;
            long long* w = sF + L.start(d, 4) + (k & 1) * L.part(d, 4) + i3[d] * L.sd(d, 4) +
                           i3[(d + 1) % 3] * L.se(d, 4) + i3[(d + 2) % 3];
            const S31 x = split31(to_fixed(__longlong_as_double(*w), k58[k]));
            *reinterpret_cast<int2*>(w) = make_int2(x.lo, x.hi);
          }
        }
      }
    }
    __syncthreads();

    // ---- gather, push, move ----
    const double dtd[3] = {g.dt / g.dx, g.dt / g.dy, g.dt / g.dz};
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
        {
          S31 wn[3][4], wh[3][4];
          int r[3], hs[3];  // cell and half-node start (0: c-2, 1: c-1) per axis
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const long long T = to_fixed(p.o[d][idx], 62);
            const bool low = T < (1LL << 61);
            spline62(T, wn[d]);
            spline62(low ? T + (1LL << 61) : T - (1LL << 61), wh[d]);
            r[d] = l[d];
            hs[d] = low ? 0 : 1;
          }
#pragma unroll 1
          for (int d = 0; d < 3; ++d) {  // axes 0, 1, 2 of the arrays: d, e, f
            // E_d sits on half nodes of d and nodes of e, f; B_e on half nodes
            // of d and f and nodes of e: the two share the weights of (d, e)
            const int sd = L.sd(d, 4), se = L.se(d, 4);
            const int2* b = reinterpret_cast<const int2*>(sF) + L.start(d, 4) + (r[0] + hs[0]) * sd + (r[1] + 1) * se + r[2];
            S31 wde[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) wde[i][j] = splitw(mul62(wh[0][i], wn[1][j]));
            const double e = fixed_to_double(gather64(b + 1, sd, se, wde, wn[2]), sc[56 + 2 * d]);
            const double m = fixed_to_double(gather64(b + L.part(d, 4) + hs[2], sd, se, wde, wh[2]), sc[57 + 2 * d]);
            E[0] = E[1], E[1] = E[2], E[2] = e;
            B[1] = B[2], B[2] = B[0], B[0] = m;  // after three turns: B_y, B_z, B_x came in that order
            const int r0 = r[0], h0 = hs[0];
            r[0] = r[1], r[1] = r[2], r[2] = r0;
            hs[0] = hs[1], hs[1] = hs[2], hs[2] = h0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const S31 v = wn[0][k], w = wh[0][k];
              wn[0][k] = wn[1][k], wn[1][k] = wn[2][k], wn[2][k] = v;
              wh[0][k] = wh[1][k], wh[1][k] = wh[2][k], wh[2][k] = w;
            }
          }
        }
        double u[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d] = p.u[d][idx];
        // relativistic Boris push
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
          double o = p.o[d][idx] + dtd[d] * u[d] * ig;
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
        key = place_moved(P, g, tl, t, l, dc, good, origin_after, xlo, xhi, pos, ent, pn.cell + dst, keys + dst);
        if (key == t) own += 1;
      }
      count_leaving(cnt_next, key, t);
    }
    __syncthreads();

    // ---- the region becomes the J tile ----
    {
      int4* z = reinterpret_cast<int4*>(smem_raw);
      const int n = (int)(so.order / 16);
      for (int i = tid; i < n; i += kPushThreads) z[i] = make_int4(0, 0, 0, 0);
    }
    __syncthreads();
    // P 2^s = q w jc run 2^s, below 2^62 by the choice of the scale; run at 2^62
    const double jc[3] = {-1.0 / (g.dt * g.dy * g.dz), -1.0 / (g.dt * g.dx * g.dz), -1.0 / (g.dt * g.dx * g.dy)};
    for (int pos = tid; pos < nch; pos += kPushThreads) {
      const unsigned ent = order[pos];
      if (ent & kCross) continue;
      int r[3];
      L.cell((ent >> 12) & 4095, r);
      const int idx = c0 + (int)(ent & 4095), dst = c0 + pos;
      const double qw = q * p.w[idx];
      long long S[3][4], D[3][4];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        long long w1[4];
        spline62(to_fixed(p.o[d][idx], 62), S[d]);
        spline62(to_fixed(pn.o[d][dst], 62), w1);
#pragma unroll
        for (int k = 0; k < 4; ++k) D[d][k] = w1[k] - S[d][k];
      }
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {  // axes 0, 1, 2 of the arrays: d, e, f
        const int sd = L.sd(d, 5), se = L.se(d, 5), lo = L.part(d, 5);
        unsigned* j = sJ + L.start(d, 5) + (r[0] + 1) * sd + (r[1] + 1) * se + r[2] + 1;  // nodes c-1 .. c+2
        S31 Pi[3];
        {
          const double cfs = qw * (d == 0 ? jc[0] : (d == 1 ? jc[1] : jc[2])) * exp2i(sc[4 + d] - 62);
          long long run = 0;
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            run += D[0][m];
            Pi[m] = split31(to_fixed(fixed_to_double(run, 0) * cfs, 0));
          }
        }
        S31 ak[4], bk[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          ak[c] = splitw((2 * S[2][c] + D[2][c]) >> 1);       // S_f + D_f / 2
          bk[c] = splitw(third62(S[2][c], D[2][c]));  // S_f / 2 + D_f / 3
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const S31 sb = splitw(S[1][b]), db = split31(D[1][b]);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            Acc31 a = acc31_init();
            acc31(a, sb, ak[c]);
            acc31(a, db, bk[c]);
            const S31 A = splitw(max(acc31_result(a), 0LL));  // A >= 0; clamps a rounding below zero
            long long X[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) X[m] = mul62(Pi[m], A);
            add_current64<3>(j + b * se + c, lo, sd, X, 3);
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
      const double qw = q * p.w[idx];
      long long S[3][5], D[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int dc = (int)((ent >> (24 + 2 * d)) & 3u) - 1;
        long long w0[4], w1[4];
        spline62(to_fixed(p.o[d][idx], 62), w0);
        spline62(to_fixed(pn.o[d][dst], 62), w1);
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
        S31 Pi[4];
        {
          const double cfs = qw * (d == 0 ? jc[0] : (d == 1 ? jc[1] : jc[2])) * exp2i(sc[4 + d] - 62);
          long long run = 0;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            run += D[0][m];
            Pi[m] = split31(to_fixed(fixed_to_double(run, 0) * cfs, 0));
          }
        }
        S31 ak[5], bk[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          ak[c] = splitw((2 * S[2][c] + D[2][c]) >> 1);
          bk[c] = splitw(third62(S[2][c], D[2][c]));
        }
#pragma unroll
        for (int b = 0; b < 5; ++b)
          if (b < n[1]) {
            const S31 sb = splitw(S[1][b]), db = split31(D[1][b]);
#pragma unroll
            for (int c = 0; c < 5; ++c)
              if (c < n[2]) {
                Acc31 a = acc31_init();
                acc31(a, sb, ak[c]);
                acc31(a, db, bk[c]);
                const S31 A = splitw(max(acc31_result(a), 0LL));
                long long X[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) X[m] = mul62(Pi[m], A);
                add_current64<4>(j + b * se + c, lo, sd, X, n[0] - 1);
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
    __syncthreads();

    // flush: a half warp per (x, y) row, the lanes along z
    {
      const int NY = tl.ty + 5, nrow = (tl.tx + 5) * NY, NZ = tl.tz + 5;
      for (int r = tid >> 4; r < nrow; r += kPushThreads / 16) {
        const int lx = r / NY, ly = r - lx * NY;
        const int gi0 = P.tabx[lx] + P.taby[ly];
        for (int lz = tid & 15; lz < NZ; lz += 16) {
          const int i3[3] = {lx, ly, lz};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const unsigned* w = sJ + L.start(d, 5) + i3[d] * L.sd(d, 5) + i3[(d + 1) % 3] * L.se(d, 5) + i3[(d + 2) % 3];
            const long long X = (long long)(((unsigned long long)w[0] << 32) | w[L.part(d, 5)]);
            if (X != 0) atomicAdd(f.c[JX + d] + gi0 + P.tabz[lz], fixed_to_double(X, sc[4 + d]));
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
