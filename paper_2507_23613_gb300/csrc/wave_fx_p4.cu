// The fixed-point 2D step kernel instantiated for 9 to 11 frequencies.
#include "wave_fx_kernels.cuh"

namespace mfwh {

FxFn fx_fn_p4(int nf) {
  switch (nf) {
    case 9: return fx_launch_nf<9>;
    case 10: return fx_launch_nf<10>;
    default: return fx_launch_nf<11>;
  }
}

}  // namespace mfwh
