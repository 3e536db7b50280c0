// make_eos_fix of a derived EOS block as a caller of pplbm_step_noalloc hands it in, for the
// CPU tests: prints ok and loop of the fixed-point factors. Arguments: mode, b, G, rho_v,
// rho_max, rho_min, rho_l, p_max, p_min, a1sq, a3sq.
#include <cstdio>
#include <cstdlib>

#include "../../paper_2107_06355_gb300/csrc/collision_args.cpp"

int main(int argc, char** argv) {
  if (argc != 12) return 2;
  double v[11];
  for (int i = 0; i < 11; ++i) v[i] = std::strtod(argv[1 + i], nullptr);
  pplbm_eos_derived d{};
  d.mode = (int32_t)v[0];
  d.b = v[1];
  d.G = v[2];
  d.rho_v = v[3];
  d.rho_max = v[4];
  d.rho_min = v[5];
  d.rho_l = v[6];
  d.p_max = v[7];
  d.p_min = v[8];
  d.a1sq = v[9];
  d.a3sq = v[10];
  d.b1 = d.b3 = 1e-3;
  const pplbm::EosFix e = pplbm::make_eos_fix(d, v[2]);
  std::printf("%d %d\n", e.ok, e.loop);
  return 0;
}
