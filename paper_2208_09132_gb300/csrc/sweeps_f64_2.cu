// sweeps_f64_2.cu -- the FP64 tile shapes of the CDUGKS step for D = 2.
#include "sweeps_impl.cuh"

namespace cdg {

namespace {
[[maybe_unused]] constexpr int FF = MODE_FUSED | MODE_FACES, SF = MODE_STORED | MODE_FACES, FG = FF | MODE_R2;
[[maybe_unused]] constexpr int FFS = FF | MODE_SK, SFS = SF | MODE_SK;   // Shakhov collision
[[maybe_unused]] constexpr int PFA = MODE_PREP | MODE_FACES | MODE_ACC;   // external acceleration
using List = ShapeList<Shape<double, 2, 16, 8, 1>, Shape<double, 2, 8, 8, 1>, Shape<double, 2, 16, 8, 1, MODE_STORED>,
                       Shape<double, 2, 16, 8, 1, FF>, Shape<double, 2, 8, 8, 1, FG>, Shape<double, 2, 16, 8, 1, FFS>,
                       Shape<double, 2, 16, 8, 1, PFA>, LeanShape<double, 2, 16, 8, 1>>;
}  // namespace

const ShapeOps<double>& shapes_f64_2() {
    static const ShapeOps<double> ops = ops_of<double, List>();
    return ops;
}

}  // namespace cdg
