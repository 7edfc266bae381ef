// sweeps_f32_1.cu -- the FP32-storage tile shapes of the CDUGKS step for D = 1.
#include "sweeps_impl.cuh"

namespace cdg {

namespace {
[[maybe_unused]] constexpr int FF = MODE_FUSED | MODE_FACES, SF = MODE_STORED | MODE_FACES, FG = FF | MODE_R2;
[[maybe_unused]] constexpr int FFS = FF | MODE_SK, SFS = SF | MODE_SK;   // Shakhov collision
[[maybe_unused]] constexpr int PFA = MODE_PREP | MODE_FACES | MODE_ACC;   // external acceleration
using List = ShapeList<Shape<float, 1, 256, 1, 1>, Shape<float, 1, 128, 1, 1>, Shape<float, 1, 64, 1, 1>,
                       Shape<float, 1, 256, 1, 1, FF, true>, Shape<float, 1, 256, 1, 1, FG>, Shape<float, 1, 256, 1, 1, FFS>,
                       Shape<float, 1, 256, 1, 1, PFA>, Shape<float, 1, 128, 1, 1, FF, true>, Shape<float, 1, 64, 1, 1, FF, true>>;
}  // namespace

const ShapeOps<float>& shapes_f32_1() {
    static const ShapeOps<float> ops = ops_of<float, List>();
    return ops;
}

}  // namespace cdg
