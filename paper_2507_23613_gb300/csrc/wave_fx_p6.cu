// The fixed-point 2D step kernel instantiated for 15 to 16 frequencies.
#include "wave_fx_kernels.cuh"

namespace mfwh {

FxFn fx_fn_p6(int nf) {
  switch (nf) {
    case 15: return fx_launch_nf<15>;
    default: return fx_launch_nf<16>;
  }
}

}  // namespace mfwh
