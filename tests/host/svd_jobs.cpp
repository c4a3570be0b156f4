// Which CTAs take which Jacobi SVD jobs (csrc/h2_kernels.h).
#include "../../paper_2403_01566_gb300/csrc/h2_kernels.h"

extern "C" int cta_takes(int cols, int threads) { return h2::svd_cta_takes(cols, threads); }
extern "C" int small_job(int rows, int cols) { return h2::svd_need_doubles(rows, cols) <= h2::SVD_SMALL_DOUBLES; }
