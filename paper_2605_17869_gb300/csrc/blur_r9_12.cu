// Level blur instances of radii 9 to 12 (blur.cuh).
#include "blur.cuh"

namespace sift {

BlurFn blur_r9_12(int R, int variant) {
  switch (R) {
    case 9: return blur_instance<9>(variant);
    case 10: return blur_instance<10>(variant);
    case 11: return blur_instance<11>(variant);
    default: return blur_instance<12>(variant);
  }
}

}  // namespace sift
