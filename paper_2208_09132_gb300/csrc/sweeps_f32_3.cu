// sweeps_f32_3.cu -- the FP32-storage tile shapes of the CDUGKS step for D = 3.
#include "sweeps_impl.cuh"

namespace cdg {

namespace {
[[maybe_unused]] constexpr int FF = MODE_FUSED | MODE_FACES, SF = MODE_STORED | MODE_FACES, FG = FF | MODE_R2;
[[maybe_unused]] constexpr int FFS = FF | MODE_SK, SFS = SF | MODE_SK;   // Shakhov collision
[[maybe_unused]] constexpr int PFA = MODE_PREP | MODE_FACES | MODE_ACC;   // external acceleration
using List = ShapeList<Shape<float, 3, 8, 4, 4>, Shape<float, 3, 8, 8, 4, MODE_PREP>, Shape<float, 3, 8, 8, 4, MODE_STORED>,
                       Shape<float, 3, 8, 4, 4, MODE_STORED>, Shape<float, 3, 8, 8, 4, SF>, Shape<float, 3, 8, 4, 4, SF>,
                       Shape<float, 3, 8, 8, 4, SFS>, Shape<float, 3, 8, 4, 4, PFA>, LeanShape<float, 3, 8, 8, 4>,
                       LeanShape<float, 3, 8, 4, 4>, LeanShape<float, 3, 8, 8, 4, false>>;
}  // namespace

const ShapeOps<float>& shapes_f32_3() {
    static const ShapeOps<float> ops = ops_of<float, List>();
    return ops;
}

}  // namespace cdg
