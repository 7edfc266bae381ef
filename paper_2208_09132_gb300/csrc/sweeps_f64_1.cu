// sweeps_f64_1.cu -- the FP64 tile shapes of the CDUGKS step for D = 1.
#include "sweeps_impl.cuh"

namespace cdg {

namespace {
[[maybe_unused]] constexpr int FF = MODE_FUSED | MODE_FACES, SF = MODE_STORED | MODE_FACES, FG = FF | MODE_R2;
[[maybe_unused]] constexpr int FFS = FF | MODE_SK, SFS = SF | MODE_SK;   // Shakhov collision
[[maybe_unused]] constexpr int PFA = MODE_PREP | MODE_FACES | MODE_ACC;   // external acceleration
using List = ShapeList<Shape<double, 1, 256, 1, 1>, Shape<double, 1, 128, 1, 1>, Shape<double, 1, 64, 1, 1>,
                       Shape<double, 1, 128, 1, 1, FF>, Shape<double, 1, 128, 1, 1, FG>, Shape<double, 1, 128, 1, 1, FFS>,
                       Shape<double, 1, 128, 1, 1, PFA>, Shape<double, 1, 64, 1, 1, FF, true>, Shape<double, 1, 32, 1, 1, FF>>;
}  // namespace

const ShapeOps<double>& shapes_f64_1() {
    static const ShapeOps<double> ops = ops_of<double, List>();
    return ops;
}

}  // namespace cdg
