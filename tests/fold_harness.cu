// Host-only harness of the folded full-grid sums (no device call): the chunks
// and tables that the preparation code plans, as JSON.
//
//   fold_harness plan F_MIN F_MAX DF TC_LO TC_HI DELAY (LO HI)x6
//     a prior box (Mc q chi1 chi2 L1 L2; LO == HI: fixed), t_c range and one
//     detector DELAY light seconds from the Earth's centre
//   fold_harness coeffs MC Q CHI1 CHI2 L1 L2   phase-basis coefficients
#include "../paper_2607_28265_gb300/csrc/capi.cu"

#include <cstdlib>

int main(int argc, char** argv) {
  if (argc == 8 && std::string(argv[1]) == "coeffs") {
    double cc[NBASIS];
    taylorf2_basis_coeffs(std::atof(argv[2]), std::atof(argv[3]), std::atof(argv[4]), std::atof(argv[5]),
                          std::atof(argv[6]), std::atof(argv[7]), cc);
    for (int j = 0; j < NBASIS; ++j) std::printf("%s%.17g", j ? ", " : "[", cc[j]);
    std::printf("]\n");
    return 0;
  }
  if (argc != 20 || std::string(argv[1]) != "plan") return 2;
  swig_ctx c;
  if (swig_set_grid(&c, std::atof(argv[2]), std::atof(argv[3]), std::atof(argv[4])) != SWIG_OK) return 3;
  c.prior_set = true;
  for (int i = 0; i < 6; ++i) {
    const double lo = std::atof(argv[8 + 2 * i]), hi = std::atof(argv[9 + 2 * i]);
    c.params[i] = swig_param{SWIG_PRIOR_UNIFORM, lo, hi, lo == hi ? SWIG_MODE_FIXED : SWIG_MODE_SAMPLE, lo, 0};
  }
  c.params[11] = swig_param{SWIG_PRIOR_UNIFORM, std::atof(argv[5]), std::atof(argv[6]), SWIG_MODE_SAMPLE, 0.0, 1};
  c.vertex[0][0] = std::atof(argv[7]) * kCSI;
  std::vector<FoldChunk> ck;
  std::vector<float> tab;
  fold_plan(&c, 1, ck, tab);
  const std::vector<float2> x = fold_abscissae();
  std::printf("{\"n_bins\": %lld, \"k_min\": %lld, \"rows\": %d, \"chunks\": [", (long long)c.n_bins, (long long)c.k_min,
              (int)FR_ROWS);
  for (size_t q = 0; q < ck.size(); ++q)
    std::printf("%s[%d, %d, %d, %.17g]", q ? ", " : "", ck[q].k0, ck[q].nbins, ck[q].kind, ck[q].slope_h);
  std::printf("], \"table\": [");
  for (size_t q = 0; q < tab.size(); ++q) std::printf("%s%.9g", q ? ", " : "", tab[q]);
  std::printf("], \"x\": [");
  for (size_t q = 0; q < x.size(); ++q) std::printf("%s[%.9g, %.9g]", q ? ", " : "", x[q].x, x[q].y);
  std::printf("]}\n");
  return 0;
}
