// The one-launch Daubechies-4 transforms (wavelet.cuh), a translation unit of
// its own for the build's parallelism.
#include "wavelet.cuh"

namespace firls {

bool wcl_launch_db4(int n, int R, const WclArgs& a) { return wcl_launch_kind<2>(n, R, a); }
int wcl_wide_db4(int n) { return wcl_wide_kind<2>(n); }
bool wcl_prepare_db4() { return wcl_attrs_kind<2>(); }

}  // namespace firls
