// Level blur instances of radii 5 to 8 (blur.cuh).
#include "blur.cuh"

namespace sift {

BlurFn blur_r5_8(int R, int variant) {
  switch (R) {
    case 5: return blur_instance<5>(variant);
    case 6: return blur_instance<6>(variant);
    case 7: return blur_instance<7>(variant);
    default: return blur_instance<8>(variant);
  }
}

}  // namespace sift
