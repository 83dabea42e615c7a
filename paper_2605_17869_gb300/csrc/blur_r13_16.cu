// Level blur instances of radii 13 to 16 (blur.cuh).
#include "blur.cuh"

namespace sift {

BlurFn blur_r13_16(int R, int variant) {
  switch (R) {
    case 13: return blur_instance<13>(variant);
    case 14: return blur_instance<14>(variant);
    case 15: return blur_instance<15>(variant);
    default: return blur_instance<16>(variant);
  }
}

}  // namespace sift
