// The fixed-point 2D step kernel instantiated for 4 to 6 frequencies.
#include "wave_fx_kernels.cuh"

namespace mfwh {

FxFn fx_fn_p2(int nf) {
  switch (nf) {
    case 4: return fx_launch_nf<4>;
    case 5: return fx_launch_nf<5>;
    default: return fx_launch_nf<6>;
  }
}

}  // namespace mfwh
