// The fixed-point 2D step kernel instantiated for 12 to 14 frequencies.
#include "wave_fx_kernels.cuh"

namespace mfwh {

FxFn fx_fn_p5(int nf) {
  switch (nf) {
    case 12: return fx_launch_nf<12>;
    case 13: return fx_launch_nf<13>;
    default: return fx_launch_nf<14>;
  }
}

}  // namespace mfwh
