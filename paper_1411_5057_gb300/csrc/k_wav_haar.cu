// The one-launch Haar transforms (wavelet.cuh), a translation unit of its own
// for the build's parallelism.
#include "wavelet.cuh"

namespace firls {

bool wcl_launch_haar(int n, int R, const WclArgs& a) { return wcl_launch_kind<1>(n, R, a); }
int wcl_wide_haar(int n) { return wcl_wide_kind<1>(n); }
bool wcl_prepare_haar() { return wcl_attrs_kind<1>(); }

}  // namespace firls
