// Prints the launch plans and the split-K scratch that the engine makes for one configuration
// (arguments: tokens, dim, heads, mlp_dim, views, select_mode, topk, mlp_tokens), as one line of
// JSON.  Needs no GPU; 152 SMs.
#include "../paper_2607_12287_gb300/csrc/engine.cu"

int main(int argc, char** argv) {
  if (argc != 9) return 2;
  int a[9] = {};
  for (int i = 1; i < 9; ++i) a[i] = std::atoi(argv[i]);
  ivit_handle h;
  h.N = a[1];
  h.D = h.cfg.dim = a[2];
  h.H = h.cfg.heads = a[3];
  h.F = h.cfg.mlp_dim = a[4];
  h.SV = a[5];
  h.cfg.select_mode = a[6];
  h.cfg.topk = a[7];
  h.cfg.mlp_tokens = a[8];
  h.KPAD = 640;
  h.M_max = h.N * h.SV;
  h.num_sms = 152;
  make_plans(&h);
  auto show = [](const char* name, const GemmPlan* p, const char* end) {
    std::printf("\"%s\": [", name);
    for (int g = 0; g < kGemmSlots; ++g)
      std::printf("{\"nt\": %d, \"bn\": %d, \"splits\": %d, \"pairs\": %d, \"defer\": %d}%s", p[g].nt, p[g].bn, p[g].splits,
                  p[g].n_pairs, p[g].defer ? 1 : 0, g + 1 < kGemmSlots ? ", " : "]");
    std::printf("%s", end);
  };
  std::printf("{");
  show("full", h.plan_full, ", ");
  show("inc", h.plan_inc, ", ");
  for (int b = 0; b < h.n_bands; ++b) show(("band" + std::to_string(b)).c_str(), h.plan_band[b], ", ");
  std::printf("\"bands\": [");
  for (int b = 0; b < h.n_bands; ++b) std::printf("%s%d", b ? ", " : "", h.band_ub[b]);
  std::printf("], \"scratch\": %zu}\n", scratch_floats(&h));
  return 0;
}
