// The small-state kernel's size rule, for ctypes.
#include "../paper_2604_03816_gb300/csrc/small_fit.h"

extern "C" unsigned threads() { return svm::THREADS; }
extern "C" unsigned cluster_log2(unsigned n, unsigned max_c) { return svm::cluster_log2(n, max_c); }
extern "C" int state_fits(unsigned n, unsigned max_c) { return svm::state_fits(n, max_c); }
