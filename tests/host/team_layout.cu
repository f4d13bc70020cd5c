// team_layout.cu -- where a team keeps its adjoint arrays (coop_adjoint.cuh).
// Test infrastructure.
#include <cstring>

#include "../../paper_2312_02836_gb300/csrc/coop_adjoint.cuh"

extern "C" void layout(int n, int R, int heat, int K, int stride, int S, long long* out) {
  nb::BlobHeader h;
  std::memset(&h, 0, sizeof h);
  h.n = n;
  h.R = R;
  h.self_heating = heat;
  nb::TeamAdj a;
  nb::team_layout(h, K, stride, S, &a);
  const long long v[] = {a.lam, a.ee, a.gr, a.gt, a.mu, a.de, a.seg, a.ce, a.vs, a.total};
  std::memcpy(out, v, sizeof v);
}
