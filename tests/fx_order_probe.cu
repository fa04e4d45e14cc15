// fx_order_probe.cu -- test infrastructure: on the host, the order of the
// states in the fixed-point PIPG's padded node vectors is a permutation of
// 0 .. KS_NXB - 1, its inverse is right, and where it splits the tile, even
// rows hold nothing in odd columns.  Built by tests/test_fx_order.py once per
// model.
#include <cstdio>

#include "pdg_adjoint.cuh"

using namespace pdg;

int main() {
  constexpr FxOrder F = make_fx_order();
  int bad = 0;
  unsigned seen = 0;
  for (int p = 0; p < KS_NXB; ++p) {
    if (F.state[p] >= KS_NXB || F.place[F.state[p]] != p) ++bad;
    seen |= 1u << F.state[p];
  }
  if (seen != (1u << KS_NXB) - 1u) ++bad;
  if (F.split)
    for (int i = 0; i < NX; ++i)
      for (int c = 0; c < NX; ++c)
        if (F.place[i] % 2 == 0 && F.place[c] % 2 == 1 && stm_nz(i, c)) ++bad;
  if (!bad) std::printf("OK %d %d\n", NX, int(F.split));
  return bad;
}
