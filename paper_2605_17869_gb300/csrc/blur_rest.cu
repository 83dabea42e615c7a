// Level blur instances (blur.cuh) of the radii that the default scale space (three
// scales per octave, sigma0 1.6) does not have, 20-row tiles: a unit of its own, so
// that the usual handle loads none of it.
#include "blur.cuh"

namespace sift {

BlurFn blur_rest(int R, int variant) {
  switch (R) {
    case 1: return blur_instance<1>(variant);
    case 2: return blur_instance<2>(variant);
    case 3: return blur_instance<3>(variant);
    case 4: return blur_instance<4>(variant);
    case 6: return blur_instance<6>(variant);
    case 9: return blur_instance<9>(variant);
    case 11: return blur_instance<11>(variant);
    case 12: return blur_instance<12>(variant);
    case 14: return blur_instance<14>(variant);
    case 15: return blur_instance<15>(variant);
    default: return blur_instance<16>(variant);
  }
}

}  // namespace sift
