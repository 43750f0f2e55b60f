// The fixed-point 2D step kernel instantiated for 1 to 3 frequencies.
#include "wave_fx_kernels.cuh"

namespace mfwh {

FxFn fx_fn_p1(int nf) {
  switch (nf) {
    case 1: return fx_launch_nf<1>;
    case 2: return fx_launch_nf<2>;
    default: return fx_launch_nf<3>;
  }
}

}  // namespace mfwh
