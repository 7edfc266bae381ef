// sweeps_f64.cu -- FP64 launches of the CDUGKS step (the plain method; the tile
// shapes are instantiated in sweeps_f64_<D>.cu), plus the precision-independent
// moment kernel.
#include "sweeps_impl.cuh"

namespace cdg {

int tile_count_f64(int D) { return shapes_of<double>(D).count; }
TileShape tile_shape_f64(int D, int id) { return shapes_of<double>(D).shape(id); }
TileShape b_tile_shape_f64(int D, int id) { return shapes_of<double>(D).b_shape(id); }
int sweep_a_ctas_f64(int D, int id) { return shapes_of<double>(D).a_ctas(id); }
int sweep_b_ctas_f64(int D, int id) { return shapes_of<double>(D).b_ctas(id); }
cudaError_t prepare_shape_f64(int D, int id) { return shapes_of<double>(D).configure(id); }
size_t sweep_smem_f64(int D, int id) { return shapes_of<double>(D).smem(id); }
int tile_mode_f64(int D, int id) { return shapes_of<double>(D).mode(id); }

cudaError_t launch_step_f64(const Geo& g, const Bufs<double>& hb, const Inst<double>* in, int cur, cudaStream_t s, cudaEvent_t* ev,
                            const void* phi_in) {
    return shapes_of<double>(g.D).step(g.tile_id, g, hb, in, cur, s, ev, phi_in);
}
bool batch_persistent_f64(int D, int id) { return shapes_of<double>(D).persistent(id); }
cudaError_t launch_batch_persist_f64(int D, int id, const PHead* h, const PItem* it, const Inst<double>* in, int* cur,
                                     PState* st, int nsteps, int wait_log2, int test_hook, cudaStream_t s) {
    return shapes_of<double>(D).persist(id, h, it, in, cur, st, nsteps, wait_log2, test_hook, s);
}
cudaError_t launch_batch_step_f64(const BatchPlan& p, const Inst<double>* insts, int* cur, cudaStream_t s) {
    return run_batch_step<double>(p, insts, cur, s);
}
cudaError_t launch_init_f64(const Geo& g, const Inst<double>* in, int cur, const double* f, cudaStream_t s) {
    return run_init<double>(g, in, cur, f, s);
}
cudaError_t launch_cellc_f64(const Geo& g, const Inst<double>* in, int cur, cudaStream_t s) {
    return run_cellc<double>(g, in, cur, s);
}
cudaError_t launch_stress_f64(const Geo& g, const Inst<double>* in, int cur, double* out, cudaStream_t s) {
    return run_stress<double>(g, in, cur, out, s);
}
cudaError_t launch_finalise_f64(const Geo& g, const Inst<double>* in, int cur, cudaStream_t s) {
    return run_finalise<double>(g, in, cur, s);
}

cudaError_t launch_moments(const Geo& g, const double* W, double* out, int conserved, cudaStream_t s) {
    const unsigned blocks = (unsigned)((g.Nc + 255) / 256);
    switch (g.D) {
        case 1: k_moments<1><<<blocks, 256, 0, s>>>(g, W, out, conserved); break;
        case 2: k_moments<2><<<blocks, 256, 0, s>>>(g, W, out, conserved); break;
        default: k_moments<3><<<blocks, 256, 0, s>>>(g, W, out, conserved); break;
    }
    return cudaGetLastError();
}

}  // namespace cdg
