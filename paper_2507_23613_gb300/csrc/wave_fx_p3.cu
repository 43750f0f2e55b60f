// The fixed-point 2D step kernel instantiated for 7 to 8 frequencies.
#include "wave_fx_kernels.cuh"

namespace mfwh {

FxFn fx_fn_p3(int nf) {
  switch (nf) {
    case 7: return fx_launch_nf<7>;
    default: return fx_launch_nf<8>;
  }
}

}  // namespace mfwh
