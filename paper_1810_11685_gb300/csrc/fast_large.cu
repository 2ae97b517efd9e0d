// Compile-time Stockham propagation passes for FFT extents 1024 and 1080 (see fast_kernels.cuh).
#include "fast_kernels.cuh"
namespace qpat {
QPAT_FAST_LENGTH(1024)
QPAT_FAST_LENGTH(1080)

namespace {
template <int L>
void plan_of(int* q) {
  q[0] = SPlan<L>::Q1;
  q[1] = SPlan<L>::Q2;
  q[2] = SPlan<L>::Q3;
}
}  // namespace

void fast_plan(int L, int q[3]) {
  q[0] = q[1] = q[2] = 0;
  switch (L) {
    case 24: plan_of<24>(q); break;
    case 40: plan_of<40>(q); break;
    case 48: plan_of<48>(q); break;
    case 54: plan_of<54>(q); break;
    case 56: plan_of<56>(q); break;
    case 168: plan_of<168>(q); break;
    case 288: plan_of<288>(q); break;
    case 432: plan_of<432>(q); break;
    case 576: plan_of<576>(q); break;
    case 1024: plan_of<1024>(q); break;
    case 1080: plan_of<1080>(q); break;
    default: break;
  }
}
}  // namespace qpat
