// make_eos_fix of a derived EOS block as a caller of pplbm_step_noalloc hands it in, for the
// CPU tests: prints ok and loop of the fixed-point factors and how many of 300 densities (100
// each on the vapour branch, the loop and the liquid branch) have psi in fixed point.
// Arguments: the mode, then name=value for the fields that differ from the set-up's block
// (T_r = 0.6; zero: all of them, but b and G).
#include <cstdio>
#include <cstdlib>

#include "../../paper_2107_06355_gb300/csrc/collision_args.cpp"
#include "../../paper_2107_06355_gb300/csrc/eos_setup.cpp"

int main(int argc, char** argv) {
  if (argc < 2) return 2;
  const int mode = std::atoi(argv[1]);
  const pplbm_eos_params q{mode, 0, 0.6, 0.387, 2.0, 4.0, 1.0, mode == 1 ? 0.834 : 0.446, 0.0};
  pplbm_eos_derived s, d;
  if (pplbm_eos_setup(&q, -1.0, &s)) return 3;
  d = s;
  const struct {
    const char* name;
    double* at;
  } fields[] = {{"rho_v", &d.rho_v}, {"rho_max", &d.rho_max}, {"rho_min", &d.rho_min}, {"rho_l", &d.rho_l},
                {"p_max", &d.p_max}, {"p_min", &d.p_min},     {"a1sq", &d.a1sq},       {"a3sq", &d.a3sq},
                {"dP", &d.dP}};
  for (int i = 2; i < argc; ++i) {
    if (!std::strcmp(argv[i], "zero")) {
      std::memset(&d, 0, sizeof(d));
      d.mode = mode;
      d.b = 4.0;
      d.G = -1.0;
      continue;
    }
    const char* eq = std::strchr(argv[i], '=');
    bool found = false;
    for (const auto& f : fields)
      if (eq && std::strlen(f.name) == (size_t)(eq - argv[i]) && !std::strncmp(f.name, argv[i], eq - argv[i])) {
        *f.at = std::strtod(eq + 1, nullptr);
        found = true;
      }
    if (!found) return 4;
  }
  const pplbm::EosFix e = pplbm::make_eos_fix(d, -1.0);
  const pplbm::EosConst c = pplbm::make_eos_const(s);
  const double edge[4] = {0.5 * s.rho_v, s.rho_v, s.rho_l, 1.1 * s.rho_l};
  int in[3] = {0, 0, 0};
  for (int k = 0; k < 300; ++k) {
    const int r = k / 100;
    const double rho = edge[r] + (edge[r + 1] - edge[r]) * ((k % 100) + 0.5) / 100.0;
    const pplbm::fx::u64 b = pplbm::fx::bits_of(rho);
    pplbm::fx::i64 P;
    int ex;
    in[r] += e.ok && pplbm::psi2_fixed(e, c, pplbm::fx::significand(b), (int)(b >> 52), (pplbm::fx::i64)b, &P, &ex);
  }
  std::printf("%d %d %d %d %d\n", e.ok, e.loop, in[0], in[1], in[2]);
  return 0;
}
