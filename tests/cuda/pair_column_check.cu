// Test helper: the column choice of the interpolation's back-substitution
// (host code only), for tests/test_pair_columns_host.py.
#include "../../paper_1909_07321_gb300/csrc/dense_smem.cuh"

extern "C" int pair_column(int pair, int n_rhs) { return rmgb::pair_column(pair, n_rhs); }
