// Level blur instances (blur.cuh) of the radii of blur_rest.cu, 40-row tiles: loaded
// only by handles whose tuning asks for them.
#include "blur.cuh"

namespace sift {

BlurFn blur_rest64(int R, int variant) {
  switch (R) {
    case 1: return blur_instance64<1>(variant);
    case 2: return blur_instance64<2>(variant);
    case 3: return blur_instance64<3>(variant);
    case 4: return blur_instance64<4>(variant);
    case 6: return blur_instance64<6>(variant);
    case 9: return blur_instance64<9>(variant);
    case 11: return blur_instance64<11>(variant);
    case 12: return blur_instance64<12>(variant);
    case 14: return blur_instance64<14>(variant);
    case 15: return blur_instance64<15>(variant);
    default: return blur_instance64<16>(variant);
  }
}

}  // namespace sift
