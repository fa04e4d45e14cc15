// plain_smem_probe.cu -- test infrastructure: on the host, the shared memory
// that a plain-form launch asks for (plain_total) holds the layout of every
// kernel of that form, for every node count, control size and PIPG layout.
// Built by tests/test_plain_smem.py once per model.
#include <cstdio>

#include "pdg_adjoint.cuh"

using namespace pdg;

int main() {
  int bad = 0, cases = 0, grew = 0;
  const int nus[2] = {4, PDG_MODEL_NU_ALT};
  for (int nu : nus)
    for (int N = 2; N <= NMAX; ++N)
      // PIPG form 3: its lane groups' threads, the other kernels at least 128;
      // form 2: its threads, the other kernels at most 512
      for (int form = 2; form <= 3; ++form) {
        const int t3 = pipg_ks_threads(N) < 64 ? 64 : pipg_ks_threads(N), t2 = pipg_reg_threads(N, nu);
        const int T = form == 3 ? t3 : t2, Tr = form == 3 ? (T < 128 ? 128 : T) : (T < 512 ? T : 512);
        const int have = plain_total(N, nu, T, Tr);
        if (have > make_lay(N, nu, T).total) ++grew;
        for (int n = 2; n <= N; ++n) {
          ++cases;
          if (make_lay(n, nu, T).total > have || make_lay(n, nu, Tr).total > have) {
            if (++bad < 10) std::printf("FAIL N=%d n=%d nu=%d form %d\n", N, n, nu, form);
          }
        }
      }
  if (!bad) std::printf("OK %d %d\n", cases, grew);
  return bad != 0;
}
