// pdg_pipg_fx.cuh -- PIPG_custom of an FP64 instance in 64-bit fixed point.
#pragma once

namespace pdg {

// ---------------------------------------------------------------------------
// Why integers.  GB300 issues two FP64 FMAs a clock and SM, and 64 of the
// 32 x 32 + 64-bit integer multiply-adds (measured: 0.052 and 1.93 warp
// instructions a clock and SM), so the FP64 loop of phase_pipg is bound by
// the FP64 pipe, where three integer multiply-adds in place of one FMA cost a
// twelfth.  The iteration here has no floating-point instruction in it; the
// stop test compares in FP64.
//
// Variables.  With psi = phi / sqrt(omega), theta likewise, gamma = alpha
// sqrt(omega) and M = gamma K, the iteration of Alg. PIPG_custom reads
//   x' = c1 x~ - M^T psi~ + ...,  psi' = psi~ + M (2 x' - x~) + gamma (w + ...)
// so one matrix M of spectral norm at most one serves both steps (x and u are
// held negated: the primal step then only adds), and every iterate lives at
// one scale: 64-bit integers X in units of 2^(gb - 61) with |X| < 2^61.
//
// Products.  M is held as h 2^30 + l in units of 2^-60 (both signed, 32 bits),
// an iterate is split as h 2^31 + 2 l; h h, h l and l h are summed in two
// 64-bit accumulators, and l l (below half of the last unit) is left out.  Of
// the sum of h h and of the result only the low 64 bits count, so they may wrap
// on the way.  The cross products must not: with |X| < 2^61 their sum is below
// (s + n) 2^59 for n terms and a sum s of |M| over them, n <= 10 here, and the
// loop is not entered with an s above FX_LANE.  Nor is it where the |M| of a
// whole row or column, with the scalar terms beside it, come to more than
// FX_SUM: then a result is below 7 2^61, and one that leaves the range cannot
// wrap back into it unseen (default parameters: sums of 2.8 to 3.1).
//
// Range.  Every iterate that is multiplied or stored is or-ed into a word of
// magnitudes; every 10 iterations the CTA looks at it.  The unit follows the
// largest iterate by shifts, so that it fills the range (from a cold start it
// keeps a bit or two of headroom while the iterates grow).  A value beyond the
// range sends the loop back to the last look's state, ten iterations, at a unit
// four times as coarse: that costs less than headroom would in precision.
//
// Precision.  The rounding is absolute, about 2^-60 of the range a sum, where
// FP64's is 2^-53 of each entry: finer for whatever is within 2^-7 of the
// largest iterate, and for small entries that large ones feed (their sums
// round in FP64 at the large ones' scale).  What it could cost are groups that
// sink far below the rest, so the loop returns -1, and the caller runs the
// FP64 loop, where at the end the largest control or the largest phi is below
// 2^-8 of the range, or theta, if any is not zero, below 2^-20 of it or weighed
// against an eps below 2^-20 of it; and before the loop where a control column
// has no entry of M of 2^-12 (with a gamma below 2^-24 the controls hardly move).
// Default parameters stay within 2^-6.9, 2^-4 and 2^-8.7 (controls, phi,
// columns), and theta sends about one in 10 000 of their loops to FP64.
// Likewise where the data is not finite, an entry of M above 1.2 shows that the
// power iteration fell short, or the iterates grow 2^40 past the data.
//
// Errors against 80-bit arithmetic in x_hat, u_hat, phi and theta, relative to
// each array's largest, root mean square over the subproblems of SCP iterations
// 1 to 9 of dispersed solves with N = 6 to 32 (1344, 768 and 768 of them; the
// FP64 loop's in brackets; emulated on the host):
//   6-DoF nu = 4    20   2.7e-16 (2.2e-15)  3.0e-16 (8.0e-16)  1.4e-16 (2.6e-16)  4.9e-15 (8.1e-15)
//                  200   5.1e-16 (5.6e-15)  5.0e-16 (4.5e-15)  1.6e-16 (1.6e-15)  1.8e-15 (2.9e-15)
//                 2000   3.7e-15 (4.6e-14)  3.1e-15 (4.0e-14)  6.3e-16 (1.6e-14)  6.3e-15 (3.0e-14)
//   6-DoF nu = 7    20   6.5e-16 (5.2e-15)  6.8e-16 (7.9e-16)  2.2e-16 (2.4e-16)  1.0e-15 (2.1e-15)
//                 2000   8.9e-16 (8.6e-15)  5.8e-16 (1.7e-15)  3.6e-16 (1.5e-15)  1.8e-14 (1.4e-14)
//   3-DoF           20   9.8e-16 (1.1e-14)  3.6e-16 (6.1e-16)  1.3e-16 (2.3e-16)  3.4e-16 (2.8e-15)
//                 2000   9.8e-16 (1.3e-14)  4.3e-16 (8.1e-16)  1.7e-16 (5.6e-16)  5.0e-16 (2.2e-15)
// The virtual controls (w_ep 0.3 to 100): 1.0 to 8.4e-16 (3.6e-16 to 1.3e-14).
// What stays behind are thetas far below phi: one in a thousand by about 5
// times, more where P_x takes y far from the other states.
//
// Work split: the tiles and butterflies of phase_pipg_ks.  At N = 15 a CTA
// runs 128 threads and about 4200 warp instructions an iteration, 900 of them
// multiply-adds, against 382 FP64 instructions of 16 cycles each.  Measured
// (4096 instances, N = 15): 31.6 ms per 1000 iterations, 2420 cycles an
// instance and iteration against 6890 of phase_pipg; N = 30 (1024 instances)
// 16.0 ms; one instance alone 1.76 us an iteration (N = 10).  Bound by latency
// and issue: two CTAs (8 warps) an SM at 255 registers, 1.4 instructions a
// clock; a third CTA at 168 registers adds spills and no speed.
// ---------------------------------------------------------------------------
struct FxM { int h, l; };  // matrix entry: (h 2^30 + l) 2^-60
struct FxC { int h, l2; };  // constant: (h 2^30 + l2 / 2) 2^-60
struct FxR { int h, l; };   // relaxation less one: (h 2^31 + l) 2^-62
struct FxV { int h, l; };  // iterate: h 2^31 + 2 l
struct FxAcc {
  long long hh = 0, cr = 1LL << 28;  // cr: rounds the shift of fx_fin
};

// c + a b; written out because the compiler widens loop-invariant factors
// ahead of the loop and then multiplies 64 by 64 bits (4100 cycles an instance
// and iteration against 2580 in the first version of this loop)
__device__ __forceinline__ long long fx_mw(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ int fx_low31(long long x) { return int(unsigned(x) << 1) >> 1; }
__device__ __forceinline__ int fx_high(long long x, int l31) { return int(x >> 31) + int(unsigned(l31) >> 31); }
__device__ __forceinline__ FxV fx_split(long long x) {
  const int l = fx_low31(x);
  return FxV{fx_high(x, l), (l + 1) >> 1};
}
__device__ __forceinline__ void fx_mad(FxAcc& a, FxM m, FxV v) {
  a.hh = fx_mw(m.h, v.h, a.hh);
  a.cr = fx_mw(m.h, v.l, a.cr);
  a.cr = fx_mw(m.l, v.h, a.cr);
}
__device__ __forceinline__ long long fx_fin(const FxAcc& a) { return (a.hh << 1) + (a.cr >> 29); }
// x c, for |x| < 2^62 and 0 <= c < 2
__device__ __forceinline__ long long fx_mul(long long x, FxC c) {
  const int l = fx_low31(x), h = fx_high(x, l);
  const long long cr = fx_mw(h, c.l2, fx_mw(l, c.h, 1LL << 29));
  return (fx_mw(h, c.h, 0) << 1) + (cr >> 30);
}
__device__ __forceinline__ FxC fx_const(long long c) {
  const int l = int(unsigned(c) << 2) >> 2;
  return FxC{int((c - l) >> 30), 2 * l};
}
__device__ __forceinline__ FxM fx_entry(long long m) {
  const int l = int(unsigned(m) << 2) >> 2;
  return FxM{int((m - l) >> 30), l};
}
// x + (rho - 1) e: the relaxed iterate from the new one and its step
__device__ __forceinline__ long long fx_relax(long long x, long long e, FxR r) {
  const int l = fx_low31(e), h = fx_high(e, l);
  return fx_mw(h, r.h, x) + (fx_mw(h, r.l, fx_mw(l, r.h, 1LL << 30)) >> 31);
}
// a b s to the nearest integer, a = ah + al, s a power of two
__device__ __forceinline__ long long fx_prod(double ah, double al, double b, double s) {
  const double bs = b * s, p = ah * bs;
  return __double2ll_rn(p) + __double2ll_rn(fma(al, bs, fma(ah, bs, -p)));
}
__device__ __forceinline__ long long fx_sat(long long x) {
  constexpr long long m = 1LL << 62;
  return x > m ? m : (x < -m ? -m : x);
}
__device__ __forceinline__ unsigned fx_mag(long long x) {
  const int h = int(x >> 32);
  return unsigned(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned long long fx_abs(long long x) { return (unsigned long long)(x < 0 ? -x : x); }
__device__ __forceinline__ long long fx_max0(long long x) { return x < 0 ? 0 : x; }
// x 2^-s to the nearest integer (s > 0), or x 2^-s exactly (s <= 0)
__device__ __forceinline__ long long fx_shift(long long x, int s) {
  return s > 0 ? (x + (1LL << (s - 1))) >> s : (long long)((unsigned long long)x << -s);
}
__device__ __forceinline__ unsigned block_or(unsigned v, unsigned* red) {
  const int nw = (blockDim.x + 31) >> 5;
  v = __reduce_or_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned m = 0;
  for (int i = 0; i < nw; ++i) m |= red[i];
  __syncthreads();
  return m;
}

// Order of the states in the padded node vector.  A lane's stored rows 2 h
// run over the even places of its tile, its stored columns 2 q over the even
// ones too (ks_perm flips only higher bits).  So where half of the states
// depend on nothing outside that half (6-DoF: mass, attitude and rates; 3-DoF:
// mass and velocity), they take the even places, and a quarter of every
// lane's tile, even rows times odd columns, is structurally zero: it is
// neither held nor multiplied (16 of 96 tile registers, 48 of 288
// multiply-adds).  Other models, and those with fewer states than half of the
// places, keep their order and the whole tile.
struct FxOrder {
  unsigned char state[KS_NXB], place[KS_NXB];  // state NX and up: padding
  bool split;
};
__host__ __device__ constexpr FxOrder make_fx_order() {
  FxOrder F{};
  const StmOrder S = make_stm_order();
  unsigned even = 0;
  F.split = NX >= KS_NXB / 2;
  for (int a = 0; F.split && a < KS_NXB / 2; ++a) even |= 1u << S.row_order[NX - 1 - a];  // the sparsest rows
  for (int a = 0; F.split && a < KS_NXB / 2; ++a) F.split = (S.row_mask[S.row_order[NX - 1 - a]] & ~even) == 0;
  int e = 0, o = 1;
  for (int i = 0; i < KS_NXB; ++i) {
    int p = i;
    if (F.split) {
      if (i < NX && ((even >> i) & 1u)) { p = e; e += 2; } else { p = o; o += 2; }
    }
    F.state[p] = (unsigned char)i;
    F.place[i] = (unsigned char)p;
  }
  return F;
}
static __constant__ FxOrder kFx = make_fx_order();
constexpr bool FX_SPLIT = make_fx_order().split;
constexpr int FX_IY = make_fx_order().place[IY], FX_IM = make_fx_order().place[IM];
__host__ __device__ constexpr bool fx_zero(int s, int q) { return FX_SPLIT && (s & 1) == 0 && (q & 1) == 1; }

// The exchange region, behind everything make_lay lays out (64-bit elements,
// 16-byte aligned rows, states by their place): psi~ and 2 x - x~ (split) and gamma w of every interval
// or node [N][KS_NXB], 2 u - u~ (split) and the control gradients [N][nup],
// gamma theta~, gamma eps [N], the dilation box and, behind it, no box [N + 1], the fixed components of the
// first and the last node [2][KS_NXB], alpha w_ep, alpha w_cost and zero, the
// last look (FxLook), the
// relaxed virtual controls, then the unextrapolated iterates of the stop test.
// The state at the last look (sn), a slot of `slot` entries for each lane, lies
// in the FP64 loop's scratch, which is idle meanwhile, where it fits (6-DoF and
// 3-DoF: always).
struct FxLay {
  int vp, dx, gw, du, bq, th, ep, lo, hi, zx, kc, lk, nvp, nvm, px, pu, pmp, pmm, pph, pth, sn, slot, end;
};
__host__ __device__ inline FxLay make_fx_lay(const Lay& L) {
  const int nup = KS_NC * ((L.nu + KS_NC - 1) / KS_NC), n1 = (L.N + 1) & ~1;
  FxLay Q;
  int o = (L.total + 1) & ~1;
  Q.vp = o; o += L.N * KS_NXB;
  Q.dx = o; o += L.N * KS_NXB;
  Q.gw = o; o += L.N * KS_NXB;
  Q.du = o; o += L.N * nup;
  Q.bq = o; o += L.N * nup;
  Q.th = o; o += n1;
  Q.ep = o; o += n1;
  Q.lo = o; o += n1 + 2;
  Q.hi = o; o += n1 + 2;
  Q.zx = o; o += 2 * KS_NXB;
  Q.kc = o; o += 4;
  Q.lk = o; o += 4;
  Q.nvp = o; o += L.N * KS_NXB;
  Q.nvm = o; o += L.N * KS_NXB;
  Q.px = o; o += L.N * KS_NXB;
  Q.pu = o; o += L.N * nup;
  Q.pmp = o; o += L.N * KS_NXB;
  Q.pmm = o; o += L.N * KS_NXB;
  Q.pph = o; o += L.N * KS_NXB;
  Q.pth = o; o += n1;
  Q.end = o;
  Q.slot = KS_WC + 3 * KS_WR + nup / KS_NC + 1;
  const int ns = L.N * KS_GS * Q.slot;
  Q.sn = ns <= L.red - L.img ? L.img : Q.end;
  if (Q.sn == Q.end) Q.end += ns;
  return Q;
}

// bounds on sums of |M|: over a lane's terms, over a whole row or column
constexpr double FX_LANE = 5.5, FX_SUM = 6.0;
// terms of a lane's longest sum: a tile column with x~ and the -I block, a tile
// row with the controls of both nodes and the -I block
__host__ __device__ constexpr int fx_terms(int nu) {
  const int nc = (nu + KS_NC - 1) / KS_NC, row = KS_TC + 2 * nc + 1;
  return KS_TR + 2 > row ? KS_TR + 2 : row;
}
// On fewer nodes the FP64 loop runs where gamma is below 2^-7: the intervals of
// a reference that cannot be flown on 4 or 5 nodes have blocks of up to 1e9,
// gamma falls to 1e-10, and theta's increments round away (errors of 5e-13 and
// 7e-12 against 5e-14 and 2e-14).  Nearly all SCP iterations but the first are
// so there, and whole solves take the FP64 loop's kernels at once: large batches
// are no faster in fixed point (4096 solves at N = 2 to 5, persistent form: 0.8 to
// 1.1 of the FP64 loop's rate).
constexpr int FX_NMIN = 6;
// iterations between two looks at the magnitudes
constexpr int FX_WINDOW = 10;
// the last look: its iteration and unit, the iteration before which headroom is
// kept, the parts run again so far, the coarsest unit (in shared memory: the
// loop has no registers to spare)
struct FxLook { int j, gb, hold, again, gtop; };

// Returns the iterations run (at least one), or -1 with the image untouched.
// Counts the parts run again at a coarser unit in P.loops[1].
template <int NU>
__device__ __forceinline__ int phase_pipg_fx(const DParams& P, int nodes, double sigma, int force) {
  using U = unsigned long long;
  // the layout anew from the node count: offsets that the persistent kernel
  // keeps in memory would be loaded once and then spilled around the loop
  const Lay L = make_lay(nodes, NU, blockDim.x);
  extern __shared__ __align__(16) unsigned char smraw[];
  double* const sm = reinterpret_cast<double*>(smraw);
  constexpr int NXB = KS_NXB, TR = KS_TR, TC = KS_TC, NR = KS_NR, NCB = KS_NC, GS = KS_GS;
  constexpr int WR = KS_WR, WC = KS_WC;
  static_assert(WR == 2 && WC == 2, "the lane's rows and components load as pairs");
  constexpr int NC = (NU + NCB - 1) / NCB;  // control columns per lane
  constexpr int NUP = NCB * NC;
  const int N = L.N, tid = threadIdx.x;
  const FxLay Q = make_fx_lay(L);
  long long* const ex = reinterpret_cast<long long*>(smraw);
  const int g = tid / GS, ln = tid - GS * g;
  const int rb = ln / NCB, cb = ln - NCB * rb;
  // roles of threads past the last group: see phase_pipg_ks
  const bool wlive = (tid & ~31) < N * GS;
  const bool live = g < N, has_iv = g < N - 1;
  const int gv = live ? g : N - 1;
  const int gm1 = gv > 0 ? gv - 1 : 0, gp1 = gv < N - 1 ? gv + 1 : gv;
  const int c0 = TC * cb + WC * rb;  // the lane's x components c0, c0 + 1 of node g
  const int i0 = TR * rb + WR * cb;  // the lane's dual rows i0, i0 + 1 of interval g
  const double wp = P.w_prox, om = P.omega;
  const double alpha = 2.0 / (wp + sqrt(wp * wp + 4.0 * om * sigma));
  // sqrt(omega), its inverse and gamma to twice the precision (high + low)
  const double so = sqrt(om), sol = fma(-so, so, om) / (2.0 * so);
  const double is = 1.0 / so, isl = is * (fma(-is, so, 1.0) - is * sol);
  const double ga = alpha * so, gal = fma(alpha, so, -ga) + alpha * sol;
  // ---- scales, and whether the data suits (the same answer on every thread)
  U top[3] = {0, 0, 0};  // largest constant; largest iterate; largest |M|
  unsigned cols = 0;     // control columns with an entry; with one of at least 2^-12
  {
    using OB = OrdBits<double>;
    for (int t = tid; t < (N - 1) * NX; t += blockDim.x) {
      top[0] = umax(top[0], OB::abs(ga * sm[L.w + t]));
      top[1] = umax(top[1], umax(OB::abs(is * sm[L.phi + t]), umax(OB::abs(sm[L.mup + t]), OB::abs(sm[L.mum + t]))));
    }
    for (int t = tid; t < N * NX; t += blockDim.x) top[1] = umax(top[1], OB::abs(sm[L.xh + t]));
    for (int t = tid; t < N * NU; t += blockDim.x) top[1] = umax(top[1], OB::abs(sm[L.uh + t]));
    for (int t = tid; t < N - 1; t += blockDim.x) {
      top[0] = umax(top[0], OB::abs(ga * sm[L.eps + t]));
      top[1] = umax(top[1], OB::abs(is * sm[L.th + t]));
    }
    for (int t = tid; t < NX; t += blockDim.x) top[0] = umax(top[0], umax(OB::abs(sm[L.zi + t]), OB::abs(sm[L.zf + t])));
    for (int t = tid; t < (N - 1) * STM_SAS; t += blockDim.x) top[2] = umax(top[2], OB::abs(ga * sm[L.Am + t]));
    // (the padding entry of an odd block stride is not written)
    for (int t = tid; t < (N - 1) * NX * NU; t += blockDim.x) {
      const int k = t / (NX * NU), o = k * b_stride(NU) + t - k * (NX * NU);
      const U b = umax(OB::abs(ga * sm[L.Bm + o]), OB::abs(ga * sm[L.Bp + o]));
      top[2] = umax(top[2], b);
      cols |= ((b > 0 ? 256u : 0u) | (b >= 0x3F30000000000000ull ? 1u : 0u)) << (t % NU);  // 2^-12
    }
    if (tid == 0) top[0] = umax(top[0], OB::abs(alpha * P.w_cost));
    block_max_u<U, 3>(top, reinterpret_cast<U*>(sm + L.red));
    cols = block_or(cols, reinterpret_cast<unsigned*>(sm + L.red));
  }
  const double vc = __longlong_as_double((long long)top[0]), vs = __longlong_as_double((long long)top[1]);
  const double mx = __longlong_as_double((long long)top[2]);
  // The unit follows the data.  w_ep is no iterate: alpha w_ep saturates (see
  // below), so a large one must not coarsen the unit of everything else (with
  // it, x_hat after 20 iterations was off by 3.4e-11 at w_ep = 1e6 and 0.36 at
  // 1e16, relative to its largest; without it by 3e-16).
  const double ref = fmax(vc, vs);
  // the range test of |M|: sigma bounds its spectral norm by one; an entry over
  // 1.2 shows that the power iteration fell short
  if (!(mx <= 1.2 && vc < 1e60 && vs < 1e60 && ref > 1e-60 && ga > 0.0 && ga <= 1.2 && P.rho > 0.0 && P.rho < 1.99 &&
        alpha * wp < 1.0 && P.w_ep >= 0.0 && P.w_ep < 1e60 && (((cols >> 8) & ~cols & 255u) == 0 || ga < 0x1p-24) &&
        (nodes >= FX_NMIN || ga >= 0x1p-7)))
    return -1;
  const int gmin = ilogb(fmax(vc, 1e-60)) + 2;  // unit bound: constants below half of the range
  const FxC GM = fx_const(fx_prod(ga, gal, 1.0, 0x1p60));
  FxR RL;
  {
    const long long c = __double2ll_rn((P.rho - 1.0) * 0x1p62);
    RL.l = fx_low31(c);
    RL.h = int((c - RL.l) >> 31);
  }
  // ---- tiles of M, in the lane's stored order (see ks_perm)
  const int prow = ks_perm<NCB, TR>(cb), pcol = ks_perm<NR, TC>(rb);
  FxM ap[TR][TC], bm[TR][NC], bp[TR][NC];
  auto entry = [&](bool ok, int off) {
    return fx_entry(ok ? fx_prod(ga, gal, sm[off], 0x1p60) : 0);
  };
#pragma unroll
  for (int s = 0; s < TR; ++s) {
    const int r = kFx.state[TR * rb + (s ^ prow)];
#pragma unroll
    for (int q = 0; q < TC; ++q) {
      if (fx_zero(s, q)) { ap[s][q] = FxM{0, 0}; continue; }
      const int c = kFx.state[TC * cb + (q ^ pcol)];
      const bool ok = has_iv && r < NX && c < NX;
      ap[s][q] = entry(ok, ok ? L.Am + g * STM_SAS + stm_index(r, c) : 0);
    }
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const int cc = cb + NCB * q;
      const bool ok = has_iv && r < NX && cc < NU;
      const int o = ok ? g * b_stride(NU) + r * NU + cc : 0;
      bm[s][q] = entry(ok, L.Bm + o);
      bp[s][q] = entry(ok, L.Bp + o);
    }
  }
  // scalar entries, zero on the lanes of groups that hold no such quantity:
  // 1 - alpha w_prox for x~ and (on the first tile row) u~, gamma for the -I
  // blocks next to hat A^-
  const long long c1 = (1LL << 60) - fx_prod(alpha, 0.0, wp, 0x1p60), g1 = fx_prod(ga, gal, 1.0, 0x1p60);
  const FxM cx1 = fx_entry(live ? c1 : 0), cu1 = fx_entry(live && rb == 0 ? c1 : 0);
  const FxM gxm = fx_entry(live ? -g1 : 0), gdm = fx_entry(has_iv ? -g1 : 0);
  {  // the sums of |M|, in units of 2^-26 and rounded up
    static_assert(FX_LANE + fx_terms(NU) < 16.0, "the cross products' accumulator");
    auto mag = [](FxM m) { return (unsigned(m.h < 0 ? -m.h : m.h) >> 4) + 1u; };
    const unsigned gm = mag(fx_entry(g1)), cm = mag(fx_entry(c1));
    unsigned sum[4] = {0, 0, 0, 0};  // of a lane; rows and x columns; control columns of hat B^- and hat B^+
    if (wlive) {
      unsigned row[TR], rs[WR], col[TC], cs[WC];
#pragma unroll
      for (int q = 0; q < TC; ++q) col[q] = 0;
#pragma unroll
      for (int s = 0; s < TR; ++s) {
        row[s] = 0;
#pragma unroll
        for (int q = 0; q < TC; ++q) { row[s] += mag(ap[s][q]); col[q] += mag(ap[s][q]); }
#pragma unroll
        for (int q = 0; q < NC; ++q) row[s] += mag(bm[s][q]) + mag(bp[s][q]);
        sum[0] = umax(sum[0], row[s] + gm);
      }
#pragma unroll
      for (int q = 0; q < TC; ++q) sum[0] = umax(sum[0], col[q] + cm + gm);
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        unsigned m = 0, p = 0;
#pragma unroll
        for (int s = 0; s < TR; ++s) { m += mag(bm[s][q]); p += mag(bp[s][q]); }
        sum[0] = umax(sum[0], umax(m + cm, p));
        sum[2] = umax(sum[2], ks_all_sum<NR, NCB>(m));
        sum[3] = umax(sum[3], ks_all_sum<NR, NCB>(p));
      }
      ks_reduce_scatter<NCB, 1>(row, rs);
      ks_reduce_scatter<NR, NCB>(col, cs);
      // (theta enters a column twice, the constants up to half of the range)
#pragma unroll
      for (int e = 0; e < WR; ++e) sum[1] = umax(sum[1], rs[e] + gm);
#pragma unroll
      for (int e = 0; e < WC; ++e) sum[1] = umax(sum[1], cs[e] + cm + 3 * gm + (1u << 25));
    }
    block_max_u<unsigned, 4>(sum, reinterpret_cast<unsigned*>(sm + L.red));
    constexpr unsigned top_sum = unsigned(FX_SUM * 0x1p26);
    if (sum[0] > unsigned(FX_LANE * 0x1p26) || sum[1] > top_sum || sum[2] + sum[3] + cm > top_sum) return -1;
  }
  bool fx[WC];
#pragma unroll
  for (int e = 0; e < WC; ++e) {
    const int c = kFx.state[c0 + e];
    fx[e] = live && c < NX && (g == 0 || (g == N - 1 && P.fix_f[c]));
  }
  const bool okx[WC] = {live && kFx.state[c0] < NX, live && kFx.state[c0 + 1] < NX};
  const bool okd[WR] = {has_iv && kFx.state[i0] < NX, has_iv && kFx.state[i0 + 1] < NX};
  const bool th_lane = has_iv && FX_IY >= i0 && FX_IY < i0 + WR;
  // where the lane finds what most lanes do not have (then a zero): the CTCS
  // duals of its y component, the cost of its mass, its dilation box
  const bool y_lane = live && FX_IY >= c0 && FX_IY < c0 + WC;
  const int tha = y_lane ? gm1 : N - 1, thb = y_lane ? gv : N - 1;
  const int kcm = (g == N - 1 && FX_IM >= c0 && FX_IM < c0 + WC) ? 1 : 2;
  const int box = cb + NCB * (NC - 1) == NU - 1 ? gv : N;
  const int gq = live ? g : 0;  // (node 1 has no control gradient from before it)
  const int jmax = force > 0 ? force : P.pipg_jmax;
  const bool chk_on = force <= 0 && P.pipg_jcheck > 0;
  const int per = chk_on ? P.pipg_jcheck : jmax;
  // A part that leaves the range is run again from the last look's state.  With
  // a stop test in every iteration that would need the unextrapolated iterates
  // of the look as well; such a loop starts anew, and keeps its unit.
  const bool roll = per > 1;
  // range 4 to 8 times the largest quantity in sight; from a cold start, whose
  // iterates grow for some hundred iterations, 16 to 32 times and with a bit of
  // headroom kept that long (without: six parts run again, 3 % of 2000 iterations)
  const bool cold = vs == 0.0;
  int gb = ilogb(ref) + (cold ? 4 : 2);
  FxLook* const look = reinterpret_cast<FxLook*>(ex + Q.lk);
  if (tid == 0) *look = FxLook{0, gb, cold ? 300 : 0, 0, gb + 40};  // past gtop the iteration diverges
  __syncthreads();
  for (; gb <= look->gtop; gb += 2) {
    if (gb < gmin) gb = gmin;
    double sc = ldexp(1.0, 61 - gb);
    long long xt[WC], ft[WR], ut[NC], tht = 0;
    FxV fg[TR];
    unsigned psi_t = 0;  // |psi| below this (in units of 2^32) leaves virtual controls of zero at zero
    // constants in the current unit.  alpha w_ep and the box saturate at twice the
    // range, beyond which they decide nothing.
    auto constants = [&]() {
      const double pt = P.w_ep * is * sc;
      psi_t = pt < 0x1p62 ? unsigned((long long)pt >> 32) : 0x7fffffffu;
      psi_t = psi_t > 0 ? psi_t - 1 : 0;
      if (tid == 0) {
        ex[Q.kc] = alpha * P.w_ep * sc < 0x1p62 ? fx_prod(alpha, 0.0, P.w_ep, sc) : 1LL << 62;
        ex[Q.kc + 1] = -fx_prod(alpha, 0.0, P.w_cost, sc);
        ex[Q.kc + 2] = 0;
        ex[Q.lo + N] = -(1LL << 62);
        ex[Q.hi + N] = 1LL << 62;
      }
      for (int t = tid; t < N * NXB; t += blockDim.x) {
        const int k = t / NXB, i = kFx.state[t - NXB * k];
        ex[Q.gw + t] = (k < N - 1 && i < NX) ? fx_prod(ga, gal, sm[L.w + k * NX + i], sc) : 0;
      }
      for (int t = tid; t < N; t += blockDim.x) {
        ex[Q.ep + t] = t < N - 1 ? fx_prod(ga, gal, sm[L.eps + t], sc) : 0;
        ex[Q.lo + t] = -fx_sat(__double2ll_rn(sm[L.hi + t] * sc));
        ex[Q.hi + t] = -fx_sat(__double2ll_rn(sm[L.lo + t] * sc));
      }
      for (int t = tid; t < NXB; t += blockDim.x) {
        const int i = kFx.state[t];
        ex[Q.zx + t] = i < NX ? -__double2ll_rn(sm[L.zi + i] * sc) : 0;
        ex[Q.zx + NXB + t] = i < NX ? -__double2ll_rn(sm[L.zf + i] * sc) : 0;
      }
    };
    // the state's exchanged parts: psi~ for node g+1 and on the whole tile row,
    // hat B^+^T psi~ for node g+1
    auto gather = [&]() {
      int vh[WR], vl[WR], h[TR], l[TR];
#pragma unroll
      for (int e = 0; e < WR; ++e) {
        const FxV v = fx_split(ft[e]);
        vh[e] = v.h; vl[e] = v.l;
      }
      if (live) *reinterpret_cast<int4*>(ex + Q.vp + g * NXB + i0) = make_int4(vh[0], vl[0], vh[1], vl[1]);
      ks_all_gather<NCB, 1>(vh, h);
      ks_all_gather<NCB, 1>(vl, l);
#pragma unroll
      for (int s = 0; s < TR; ++s) fg[s] = FxV{h[s], l[s]};
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        FxAcc a;
#pragma unroll
        for (int s = 0; s < TR; ++s) fx_mad(a, bp[s][q], fg[s]);
        const long long v = ks_all_sum<NR, NCB>(fx_fin(a));
        if (has_iv && rb == 0 && cb + NCB * q < NU) ex[Q.bq + (g + 1) * NUP + cb + NCB * q] = v;
      }
    };
    auto publish = [&]() {
      if (wlive) {
        gather();
        if (th_lane) ex[Q.th + g] = fx_mul(tht, GM);
      }
    };
    for (int t = Q.vp + tid; t < Q.pth + N; t += blockDim.x)
      if (t < Q.lk || t >= Q.nvp) ex[t] = 0;
    __syncthreads();
    constants();
#pragma unroll
    for (int e = 0; e < WC; ++e) {
      xt[e] = okx[e] ? -__double2ll_rn(sm[L.xh + g * NX + kFx.state[c0 + e]] * sc) : 0;
      if (okx[e]) ex[Q.px + g * NXB + c0 + e] = xt[e];
    }
#pragma unroll
    for (int e = 0; e < WR; ++e) {
      const int o = okd[e] ? g * NX + kFx.state[i0 + e] : 0;
      ft[e] = okd[e] ? fx_prod(is, isl, sm[L.phi + o], sc) : 0;
      if (okd[e]) {
        const int oe = g * NXB + i0 + e;
        ex[Q.pmp + oe] = ex[Q.nvp + oe] = __double2ll_rn(sm[L.mup + o] * sc);
        ex[Q.pmm + oe] = ex[Q.nvm + oe] = __double2ll_rn(sm[L.mum + o] * sc);
        ex[Q.pph + g * NXB + i0 + e] = ft[e];
      }
    }
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const int cc = cb + NCB * q;
      ut[q] = (live && cc < NU) ? -__double2ll_rn(sm[L.uh + g * NU + cc] * sc) : 0;
      if (live && cc < NU && rb == 0) ex[Q.pu + g * NUP + cc] = ut[q];
    }
    if (th_lane) {
      tht = fx_prod(is, isl, sm[L.th + g], sc);
      ex[Q.pth + g] = tht;
    }
    publish();
    __syncthreads();
    unsigned mag = 0;
    // the largest |psi~| of the lane's rows, and whether the warp holds a
    // virtual control that is not zero
    unsigned pm = umax(fx_mag(ft[0]), fx_mag(ft[1]));
    bool nz = false;
    if (wlive) {
      bool any = false;
#pragma unroll
      for (int e = 0; e < WR; ++e)
        any = any || (okd[e] && (ex[Q.nvp + g * NXB + i0 + e] | ex[Q.nvm + g * NXB + i0 + e]) != 0);
      nz = __any_sync(0xffffffffu, any);
    }
    // the state at a look, in the unit of then
    int j = 0;
    long long* const slot = ex + Q.sn + (live ? tid : 0) * Q.slot;
    auto save = [&]() {
      if (live) {
        long long* p = slot;
#pragma unroll
        for (int e = 0; e < WC; ++e) *p++ = xt[e];
#pragma unroll
        for (int e = 0; e < WR; ++e) {
          *p++ = ft[e];
          *p++ = ex[Q.nvp + g * NXB + i0 + e];
          *p++ = ex[Q.nvm + g * NXB + i0 + e];
        }
#pragma unroll
        for (int q = 0; q < NC; ++q) *p++ = ut[q];
        *p = tht;
      }
      if (tid == 0) { look->j = j; look->gb = gb; }
    };
    auto restore = [&](int s) {  // at a unit 2^s times that of the look
      bool any = false;
      if (live) {
        const long long* p = slot;
#pragma unroll
        for (int e = 0; e < WC; ++e) xt[e] = fx_shift(*p++, s);
#pragma unroll
        for (int e = 0; e < WR; ++e) {
          ft[e] = fx_shift(*p++, s);
          const long long a = fx_shift(*p++, s), b = fx_shift(*p++, s);
          ex[Q.nvp + g * NXB + i0 + e] = a;
          ex[Q.nvm + g * NXB + i0 + e] = b;
          any = any || (a | b) != 0;
        }
#pragma unroll
        for (int q = 0; q < NC; ++q) ut[q] = fx_shift(*p++, s);
        tht = fx_shift(*p, s);
      }
      if (wlive) nz = __any_sync(0xffffffffu, any);
    };
    if (roll) save();
    // V as in phase_pipg_ks: 0 plain, 1 stores the unextrapolated iterates,
    // 2 tests against the stored ones, then stores
    auto iterate = [&](auto v_tag) -> bool {
      constexpr int V = decltype(v_tag)::value;
      constexpr bool chk = V == 2, st = V >= 1;
      U zn = 0, zo = 0, zd = 0, rn = 0, ro = 0, rd = 0;
      FxV dxv[WC], duv[NC];
#pragma unroll
      for (int e = 0; e < WC; ++e) dxv[e] = FxV{0, 0};
#pragma unroll
      for (int q = 0; q < NC; ++q) duv[q] = FxV{0, 0};
      // ---- projected gradient step (primal)
      if (wlive) {
        long long cx[TC], gx[WC], cu[NC];
        const int4 vp = *reinterpret_cast<const int4*>(ex + Q.vp + gm1 * NXB + c0);
#pragma unroll
        for (int q = 0; q < TC; ++q) {
          FxAcc a;
#pragma unroll
          for (int s = 0; s < TR; ++s)
            if (!fx_zero(s, q)) fx_mad(a, ap[s][q], fg[s]);
          if (q < WC) {  // the sums that stay on this lane also take x~ and the -I block
            fx_mad(a, cx1, fx_split(xt[q]));
            fx_mad(a, gxm, q == 0 ? FxV{vp.x, vp.y} : FxV{vp.z, vp.w});
          }
          cx[q] = fx_fin(a);
        }
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          FxAcc a;
#pragma unroll
          for (int s = 0; s < TR; ++s) fx_mad(a, bm[s][q], fg[s]);
          fx_mad(a, cu1, fx_split(ut[q]));
          cu[q] = ks_all_sum<NR, NCB>(fx_fin(a)) + ex[Q.bq + gq * NUP + cb + NCB * q];
        }
        ks_reduce_scatter<NR, NCB>(cx, gx);
        gx[FX_IY & 1] += ex[Q.th + tha] - ex[Q.th + thb];  // th[N-1] stays zero
        gx[FX_IM & 1] += ex[Q.kc + kcm];
        int dv[2 * WC];
#pragma unroll
        for (int e = 0; e < WC; ++e) {
          const int c = c0 + e;
          long long xn = gx[e];
          if (fx[e]) xn = ex[Q.zx + (g == 0 ? 0 : NXB) + c];
          const long long st_ = xn - xt[e], d = xn + st_;
          dxv[e] = fx_split(d);
          dv[2 * e] = dxv[e].h;
          dv[2 * e + 1] = dxv[e].l;
          xt[e] = fx_relax(xn, st_, RL);
          mag |= fx_mag(xn) | fx_mag(d) | fx_mag(xt[e]);
          if constexpr (chk) {
            const long long old = okx[e] ? ex[Q.px + g * NXB + c] : 0;
            if (okx[e]) { zn = umax(zn, fx_abs(xn)); zo = umax(zo, fx_abs(old)); zd = umax(zd, fx_abs(xn - old)); }
          }
          if constexpr (st) {
            if (okx[e]) ex[Q.px + g * NXB + c] = xn;
          }
        }
        if (live) *reinterpret_cast<int4*>(ex + Q.dx + g * NXB + c0) = make_int4(dv[0], dv[1], dv[2], dv[3]);
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          const int cc = cb + NCB * q;
          const bool ok = live && cc < NU;
          long long un = cu[q];
          if (q == NC - 1) {
            const long long lo = ex[Q.lo + box], hi = ex[Q.hi + box];
            un = un < lo ? lo : un;
            un = un > hi ? hi : un;
          }
          const long long st_ = un - ut[q], d = un + st_;
          duv[q] = fx_split(d);
          if (ok && rb == 0) reinterpret_cast<FxV*>(ex)[Q.du + g * NUP + cc] = duv[q];
          ut[q] = fx_relax(un, st_, RL);
          mag |= fx_mag(un) | fx_mag(d) | fx_mag(ut[q]);
          if constexpr (chk) {
            if (ok) {
              const long long old = ex[Q.pu + g * NUP + cc];
              zn = umax(zn, fx_abs(un)); zo = umax(zo, fx_abs(old)); zd = umax(zd, fx_abs(un - old));
            }
          }
          if constexpr (st) {
            // after every lane of the tile column has read it
            __syncwarp();
            if (ok && rb == 0) ex[Q.pu + g * NUP + cc] = un;
          }
        }
      }
      __syncthreads();
      // ---- virtual controls and proportional-integral feedback (dual)
      if (wlive) {
        long long rr[TR], rs[WR];
        const int4 dn = *reinterpret_cast<const int4*>(ex + Q.dx + gp1 * NXB + i0);
        const longlong2 gw = *reinterpret_cast<const longlong2*>(ex + Q.gw + gv * NXB + i0);
        {
          int vh[WC], vl[WC], h[TC], l[TC];
#pragma unroll
          for (int e = 0; e < WC; ++e) { vh[e] = dxv[e].h; vl[e] = dxv[e].l; }
          ks_all_gather<NR, NCB>(vh, h);
          ks_all_gather<NR, NCB>(vl, l);
          FxV du1[NC];
#pragma unroll
          for (int q = 0; q < NC; ++q) du1[q] = reinterpret_cast<const FxV*>(ex)[Q.du + gp1 * NUP + cb + NCB * q];
#pragma unroll
          for (int s = 0; s < TR; ++s) {
            FxAcc a;
#pragma unroll
            for (int q = 0; q < TC; ++q)
              if (!fx_zero(s, q)) fx_mad(a, ap[s][q], FxV{h[q], l[q]});
#pragma unroll
            for (int q = 0; q < NC; ++q) { fx_mad(a, bm[s][q], duv[q]); fx_mad(a, bp[s][q], du1[q]); }
            if (s < WR) fx_mad(a, gdm, s == 0 ? FxV{dn.x, dn.y} : FxV{dn.z, dn.w});
            rr[s] = fx_fin(a);
          }
        }
        ks_reduce_scatter<NCB, 1>(rr, rs);
        long long d[WR] = {gw.x - rs[0], gw.y - rs[1]};
        long long mp[WR] = {0, 0}, mm[WR] = {0, 0};
        // the virtual controls are zero unless a defect cannot be closed
        if (nz || __any_sync(0xffffffffu, pm >= psi_t)) {
          const long long AW = ex[Q.kc];
          bool any = false;
#pragma unroll
          for (int e = 0; e < WR; ++e) {
            if (okd[e]) {
              const int o = g * NXB + i0 + e;
              long long a = ex[Q.nvp + o], b = ex[Q.nvm + o];
              const long long gf = fx_mul(ft[e], GM);
              mp[e] = fx_max0(a - AW - gf);
              mm[e] = fx_max0(b - AW + gf);
              d[e] += fx_mul((2 * mp[e] - a) - (2 * mm[e] - b), GM);
              a = fx_relax(mp[e], mp[e] - a, RL);
              b = fx_relax(mm[e], mm[e] - b, RL);
              ex[Q.nvp + o] = a;
              ex[Q.nvm + o] = b;
              any = any || (a | b) != 0;
              // held to an eighth of the range: their sum is multiplied
              const unsigned m = fx_mag(mp[e]) | fx_mag(mm[e]) | fx_mag(a) | fx_mag(b);
              mag |= m | (m << 3);
            }
          }
          nz = __any_sync(0xffffffffu, any);
        }
        pm = 0;
#pragma unroll
        for (int e = 0; e < WR; ++e) {
          const int o = g * NXB + i0 + e;
          if constexpr (chk) {
            if (okd[e]) {
              const long long op = ex[Q.pmp + o], oq = ex[Q.pmm + o];
              zn = umax(zn, umax(U(mp[e]), U(mm[e])));
              zo = umax(zo, umax(U(op), U(oq)));
              zd = umax(zd, umax(fx_abs(mp[e] - op), fx_abs(mm[e] - oq)));
            }
          }
          if constexpr (st) {
            if (okd[e]) { ex[Q.pmp + o] = mp[e]; ex[Q.pmm + o] = mm[e]; }
          }
          const long long pn = ft[e] + d[e];
          ft[e] = fx_relax(pn, d[e], RL);
          const unsigned m = fx_mag(ft[e]);
          pm = umax(pm, m);
          mag |= fx_mag(d[e]) | m;
          if constexpr (chk) {
            if (okd[e]) {
              const long long old = ex[Q.pph + o];
              rn = umax(rn, fx_abs(pn)); ro = umax(ro, fx_abs(old)); rd = umax(rd, fx_abs(pn - old));
            }
          }
          if constexpr (st) {
            if (okd[e]) ex[Q.pph + o] = pn;
          }
        }
        gather();
        if (th_lane) {
          const FxV ya = reinterpret_cast<const FxV*>(ex)[Q.dx + g * NXB + FX_IY];
          const FxV yb = reinterpret_cast<const FxV*>(ex)[Q.dx + gp1 * NXB + FX_IY];
          FxAcc a;
          fx_mad(a, gdm, yb);
          fx_mad(a, FxM{-gdm.h, -gdm.l}, ya);
          const long long tn = fx_max0(tht + fx_fin(a) - ex[Q.ep + g]);
          tht = fx_relax(tn, tn - tht, RL);
          mag |= fx_mag(tn) | fx_mag(tht);
          if constexpr (chk) {
            const long long old = ex[Q.pth + g];
            rn = umax(rn, U(tn)); ro = umax(ro, fx_abs(old)); rd = umax(rd, fx_abs(tn - old));
          }
          if constexpr (st) ex[Q.pth + g] = tn;
          ex[Q.th + g] = fx_mul(tht, GM);
        }
      }
      if constexpr (chk) {
        U w6[6] = {zn, zo, zd, rn, ro, rd};
        block_max_u<U, 6>(w6, reinterpret_cast<U*>(sm + L.red));
        const double eabs = P.eps_abs * sc, erel = P.eps_rel;
        return double(w6[2]) <= eabs + erel * double(umax(w6[0], w6[1])) &&
               so * double(w6[5]) <= eabs + erel * (so * double(umax(w6[3], w6[4])));
      } else {
        (void)zn; (void)zo; (void)zd; (void)rn; (void)ro; (void)rd;
        __syncthreads();
        return false;
      }
    };
    bool over = false;
    while (j < jmax) {
      // up to the next stop test, the next look at the magnitudes or the end
      // of the loop.  The last iteration before any of them stores the
      // iterates that a test right behind it compares with; where that test
      // would be a part of its own, it closes this one.
      const int to_test = per - j % per, to_look = FX_WINDOW - (j % per) % FX_WINDOW;
      int nb = to_test < jmax - j ? to_test : jmax - j;
      nb = to_look < nb ? to_look : nb;
      if (to_test == nb + 1 && nb < jmax - j) nb = to_test;
      const bool tested = chk_on && nb == to_test;
      bool stop = false;
      for (int k = tested ? 2 : 1; k < nb; ++k) iterate(KsTag<0>{});
      if (!tested || nb >= 2) iterate(KsTag<1>{});
      if (tested) stop = iterate(KsTag<2>{});
      const unsigned m = block_or(mag, reinterpret_cast<unsigned*>(sm + L.red));
      mag = 0;
      if (m >= (1u << 29)) {
        if (tid == 0) atomicAdd(P.loops + 1, 1ull);
        over = !roll;
        if (over) break;
        gb += 2;
        if (gb > look->gtop) return -1;
        restore(gb - look->gb);
        j = look->j;
        if (tid == 0) {
          look->again = look->again < 6 ? look->again + 1 : 6;
          look->hold = j + (FX_WINDOW << look->again);
        }
      } else {
        j += nb;
        if (stop || j >= jmax) break;
        // the largest magnitude to the top of the range, or (before hold) to
        // one or two bits below it
        const int slack = __clz(m) - 3;
        int s = slack < 1 ? 2 : (roll && slack > 2 ? 1 - slack : 0);
        if (roll && j >= look->hold) s = -slack;
        if (gb + s < gmin) s = gmin - gb;
        if (s != 0) {
          gb += s;
#pragma unroll
          for (int e = 0; e < WC; ++e) xt[e] = fx_shift(xt[e], s);
#pragma unroll
          for (int e = 0; e < WR; ++e) ft[e] = fx_shift(ft[e], s);
#pragma unroll
          for (int q = 0; q < NC; ++q) ut[q] = fx_shift(ut[q], s);
          tht = fx_shift(tht, s);
          for (int t = Q.nvp + tid; t < Q.pth + N; t += blockDim.x) ex[t] = fx_shift(ex[t], s);
        }
        if (s == 0) {
          if (roll) save();
          continue;
        }
      }
      sc = ldexp(1.0, 61 - gb);
      pm = umax(fx_mag(ft[0]), fx_mag(ft[1]));
      constants();
      publish();
      __syncthreads();
      if (roll) save();
    }
    if (over) continue;
    // whether every group of results keeps the precision that the FP64 loop's
    // own exponents would give it (see the header)
    U low[3] = {0, 0, 0};
    for (int t = tid; t < N * NUP; t += blockDim.x) low[0] = umax(low[0], fx_abs(ex[Q.pu + t]));
    for (int t = tid; t < (N - 1) * NXB; t += blockDim.x) low[1] = umax(low[1], fx_abs(ex[Q.pph + t]));
    for (int t = tid; t < N - 1; t += blockDim.x) low[2] = umax(low[2], fx_abs(ex[Q.pth + t]));
    block_max_u<U, 3>(low, reinterpret_cast<U*>(sm + L.red));
    if (low[0] < (1ull << 53) || low[1] < (1ull << 53)) return -1;
    if (low[2] != 0 && (low[2] < (1ull << 41) || P.eps_ctcs * P.Pxinv[IY] < ldexp(1.0, gb - 20))) return -1;
    // the unextrapolated iterates to the image (warm start of the next SCP iteration)
    const double un = ldexp(1.0, gb - 61);
    __syncthreads();
    for (int t = tid; t < N * NX; t += blockDim.x) sm[L.xh + t] = -double(ex[Q.px + (t / NX) * NXB + kFx.place[t % NX]]) * un;
    for (int t = tid; t < N * NU; t += blockDim.x) sm[L.uh + t] = -double(ex[Q.pu + (t / NU) * NUP + t % NU]) * un;
    for (int t = tid; t < (N - 1) * NX; t += blockDim.x) {
      const int o = (t / NX) * NXB + kFx.place[t % NX];
      sm[L.mup + t] = double(ex[Q.pmp + o]) * un;
      sm[L.mum + t] = double(ex[Q.pmm + o]) * un;
      const double f = double(ex[Q.pph + o]) * un;
      sm[L.phi + t] = fma(f, so, f * sol);
    }
    for (int t = tid; t < N - 1; t += blockDim.x) {
      const double f = double(ex[Q.pth + t]) * un;
      sm[L.th + t] = fma(f, so, f * sol);
    }
    __syncthreads();
    return j;
  }
  return -1;
}

}  // namespace pdg
