// fx_layout_probe.cu -- test infrastructure: on the host, the shared-memory
// layouts of the fixed-point PIPG (make_fx_lay) and of the discretization by
// column classes (make_disc_cols_lay) hold every region their kernels index,
// for instances of n nodes in a launch sized for N >= n, and the latter's warp
// roles give every column of every interval to one lane.  Built by
// tests/test_fx_layout.py once per model; prints "OK <cases>" or the failures.
#include <cstdio>

#include "pdg_adjoint.cuh"

using namespace pdg;

static int bad = 0;
#define CHECK(cond, ...)                                  \
  do {                                                    \
    if (!(cond)) {                                        \
      if (bad++ < 20) {                                   \
        std::printf("FAIL %s: ", #cond);                  \
        std::printf(__VA_ARGS__);                         \
        std::printf("\n");                                \
      }                                                   \
    }                                                     \
  } while (0)

static long cases = 0;

static void check_fx(int N, int nu, int T) {
  const int have = make_fx_lay(make_lay(N, nu, T)).end;
  for (int n = 2; n <= N; ++n) {
    ++cases;
    const Lay L = make_lay(n, nu, T);
    const FxLay Q = make_fx_lay(L);
    const int nup = KS_NC * ((nu + KS_NC - 1) / KS_NC), X = n * KS_NXB, V = n * nup;
    // the exchange region, behind the FP64 loop's layout
    const int reg[][2] = {{Q.vp, X}, {Q.dx, X}, {Q.gw, X}, {Q.du, V}, {Q.bq, V}, {Q.th, n}, {Q.ep, n}, {Q.lo, n + 1},
                          {Q.hi, n + 1}, {Q.zx, 2 * KS_NXB}, {Q.kc, 3}, {Q.lk, (int)(sizeof(FxLook) + 7) / 8},
                          {Q.nvp, X}, {Q.nvm, X}, {Q.px, X}, {Q.pu, V}, {Q.pmp, X}, {Q.pmm, X}, {Q.pph, X}, {Q.pth, n}};
    int o = L.total;
    for (auto& r : reg) {
      CHECK(r[0] >= o, "n=%d nu=%d T=%d offset %d", n, nu, T, r[0]);
      o = r[0] + r[1];
    }
    CHECK(o <= Q.end && Q.end <= have, "n=%d N=%d nu=%d T=%d", n, N, nu, T);
    // pairs of 64-bit entries load as 16 bytes
    CHECK(Q.vp % 2 == 0 && Q.dx % 2 == 0 && Q.gw % 2 == 0 && KS_NXB % 2 == 0, "n=%d nu=%d T=%d", n, nu, T);
    // the state at the last look: in the FP64 loop's scratch (never on the image or the reductions), or appended
    const bool in = Q.sn < L.total;
    CHECK(Q.slot == KS_WC + 3 * KS_WR + V / n / KS_NC + 1, "n=%d nu=%d T=%d", n, nu, T);
    CHECK(Q.sn >= (in ? L.img : Q.pth + n) && Q.sn + n * KS_GS * Q.slot <= (in ? L.red : Q.end), "n=%d nu=%d T=%d", n, nu, T);
    // reductions: three or six 64-bit values a warp
    CHECK(6 * (T / 32) <= L.total - L.red, "n=%d nu=%d T=%d", n, nu, T);
    CHECK(KS_GS * n <= T, "n=%d T=%d", n, T);
  }
}

#ifdef PDG_MODEL_HAS_COLUMN_CLASSES
static void check_disc(int N, int nu) {
  const int have = make_disc_cols_lay(make_lay(N, nu, 128), N).total;
  const int warps = disc_cols_warps(disc_cols_cap(N, nu), nu);
  CHECK(warps <= 16, "N=%d nu=%d", N, nu);
  for (int n = 2; n <= N; ++n) {
    ++cases;
    const Lay L = make_lay(n, nu, 128);
    const DiscColsLay D = make_disc_cols_lay(L, N);
    CHECK(D.stage == L.xh && D.sa >= 2 * (SA_A + NX * nu) + 4 * NX && D.sa % 2 == 1, "n=%d N=%d nu=%d", n, N, nu);
    CHECK(D.stage + D.cap * D.sa <= D.red && D.red + 16 <= D.total && D.total <= have, "n=%d N=%d nu=%d", n, N, nu);
    const int nw = (n - 1 + D.cap - 1) / D.cap, W = (n - 1 + nw - 1) / nw;
    CHECK(W >= 1 && W <= D.cap && W <= 32 && nw * W >= n - 1, "n=%d N=%d nu=%d", n, N, nu);
    const int U = disc_control_warps(W, nu), C = disc_class_warps(W);
    int seen[128] = {}, f = 0, j = 0, m = 0, cls = 0;
    for (int w = 0; w < warps; ++w) {
      const DiscRole r = disc_role(w, U, C);
      f += r.kind == 'F';
      j += r.kind == 'J';
      m += r.kind == 'M';
      if (r.kind == 'U') {
        CHECK(r.index >= 0 && r.index < U && !seen[r.index], "n=%d nu=%d warp %d", n, nu, w);
        seen[r.index] = 1;
      }
      if (r.kind == 'C') {
        CHECK(r.index >= 0 && r.index < C && !seen[64 + r.index], "n=%d nu=%d warp %d", n, nu, w);
        seen[64 + r.index] = 1;
        ++cls;
      }
    }
    int u = 0;
    for (int i = 0; i < 64; ++i) u += seen[i];
    CHECK(f == 1 && j == 1 && m == 1 && u == U && cls == C && 32 * U >= 2 * nu * W, "n=%d N=%d nu=%d", n, N, nu);
  }
}
#endif

// The bound on the cross products' 64-bit sum: n terms |m.h| |v.l| + |m.l| |v.h|
// with |v.l| and |m.l| <= 2^29, |v.h| <= 2^30, sum of |m.h| <= FX_LANE 2^30; and
// on a result that left the range: it must not wrap to within 2^61 of zero.
static void check_sums(int nu) {
  ++cases;
  const double cross = FX_LANE * 0x1p30 * 0x1p29 + fx_terms(nu) * 0x1p29 * 0x1p30 + 0x1p28;
  CHECK(cross < 0x1p63, "nu=%d", nu);
  // a dual row adds gamma w (half of the range) and the virtual controls (three eighths of it, times gamma <= 1.2)
  CHECK(FX_SUM * 0x1p61 + 0x1p60 + 1.2 * 3 * 0x1p58 <= 0x1p64 - 0x1p61, "nu=%d", nu);
  CHECK(KS_TR + 2 <= fx_terms(nu) && KS_TC + 2 * ((nu + KS_NC - 1) / KS_NC) + 1 <= fx_terms(nu), "nu=%d", nu);
}

int main() {
  check_sums(4);
  check_sums(PDG_MODEL_NU_ALT);
  const int nus[2] = {4, PDG_MODEL_NU_ALT};
  for (int a = 0; a < 2 && !(a == 1 && nus[1] == 4); ++a)
    for (int N = 2; N <= NMAX; ++N) {
      for (int T = pipg_ks_threads(N) < 64 ? 64 : pipg_ks_threads(N); T <= 256; T += 32) check_fx(N, nus[a], T);
#ifdef PDG_MODEL_HAS_COLUMN_CLASSES
      check_disc(N, nus[a]);
#endif
    }
  if (!bad) std::printf("OK %ld\n", cases);
  return bad != 0;
}
