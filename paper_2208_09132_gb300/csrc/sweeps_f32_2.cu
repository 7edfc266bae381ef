// sweeps_f32_2.cu -- the FP32-storage tile shapes of the CDUGKS step for D = 2.
#include "sweeps_impl.cuh"

namespace cdg {

namespace {
[[maybe_unused]] constexpr int FF = MODE_FUSED | MODE_FACES, SF = MODE_STORED | MODE_FACES, FG = FF | MODE_R2;
[[maybe_unused]] constexpr int FFS = FF | MODE_SK, SFS = SF | MODE_SK;   // Shakhov collision
[[maybe_unused]] constexpr int PFA = MODE_PREP | MODE_FACES | MODE_ACC;   // external acceleration
using List = ShapeList<Shape<float, 2, 32, 8, 1>, Shape<float, 2, 16, 8, 1>, Shape<float, 2, 32, 16, 1, MODE_PREP>,
                       Shape<float, 2, 32, 8, 1, MODE_STORED>, Shape<float, 2, 32, 16, 1, MODE_STORED>,
                       Shape<float, 2, 32, 16, 1>, Shape<float, 2, 32, 8, 1, FF, true>, Shape<float, 2, 32, 16, 1, FF>,
                       Shape<float, 2, 32, 8, 1, SF>, Shape<float, 2, 16, 8, 1, FG>, Shape<float, 2, 32, 8, 1, FFS>,
                       Shape<float, 2, 32, 8, 1, PFA>, LeanShape<float, 2, 32, 8, 1>, LeanShape<float, 2, 32, 16, 1>,
                       LeanShape<float, 2, 32, 8, 1, false>>;
}  // namespace

const ShapeOps<float>& shapes_f32_2() {
    static const ShapeOps<float> ops = ops_of<float, List>();
    return ops;
}

}  // namespace cdg
