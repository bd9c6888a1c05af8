// Test-only C shim over the triangular solves of paper_0707_0131_gb300/csrc/dense.cpp alone, for
// tests/test_host_dense_widths.py.
#include <complex>

#include "dense.h"

extern "C" void shim_chol_solve(int n, const eig::dense::cd *L, eig::dense::cd *B, int nrhs) {
    eig::dense::chol_solve(n, L, B, nrhs);
}
