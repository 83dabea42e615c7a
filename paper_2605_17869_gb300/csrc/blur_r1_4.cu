// Level blur instances of radii 1 to 4 (blur.cuh).
#include "blur.cuh"

namespace sift {

BlurFn blur_r1_4(int R, int variant) {
  switch (R) {
    case 1: return blur_instance<1>(variant);
    case 2: return blur_instance<2>(variant);
    case 3: return blur_instance<3>(variant);
    default: return blur_instance<4>(variant);
  }
}

}  // namespace sift
