// sweeps_f64_3.cu -- the FP64 tile shapes of the CDUGKS step for D = 3.
#include "sweeps_impl.cuh"

namespace cdg {

namespace {
[[maybe_unused]] constexpr int FF = MODE_FUSED | MODE_FACES, SF = MODE_STORED | MODE_FACES, FG = FF | MODE_R2;
[[maybe_unused]] constexpr int FFS = FF | MODE_SK, SFS = SF | MODE_SK;   // Shakhov collision
[[maybe_unused]] constexpr int PFA = MODE_PREP | MODE_FACES | MODE_ACC;   // external acceleration
using List = ShapeList<Shape<double, 3, 4, 4, 4>, Shape<double, 3, 8, 4, 4, MODE_PREP>, Shape<double, 3, 8, 4, 4, MODE_STORED>,
                       Shape<double, 3, 8, 4, 4, SF>, Shape<double, 3, 8, 4, 4, SFS>, Shape<double, 3, 8, 4, 4, PFA>>;
}  // namespace

const ShapeOps<double>& shapes_f64_3() {
    static const ShapeOps<double> ops = ops_of<double, List>();
    return ops;
}

}  // namespace cdg
