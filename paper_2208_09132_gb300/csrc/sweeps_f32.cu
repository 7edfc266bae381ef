// sweeps_f32.cu -- FP32-storage launches of the CDUGKS step (the tile shapes are
// instantiated in sweeps_f32_<D>.cu).
#include "sweeps_impl.cuh"

namespace cdg {

int tile_count_f32(int D) { return shapes_of<float>(D).count; }
TileShape tile_shape_f32(int D, int id) { return shapes_of<float>(D).shape(id); }
TileShape b_tile_shape_f32(int D, int id) { return shapes_of<float>(D).b_shape(id); }
int sweep_a_ctas_f32(int D, int id) { return shapes_of<float>(D).a_ctas(id); }
int sweep_b_ctas_f32(int D, int id) { return shapes_of<float>(D).b_ctas(id); }
cudaError_t prepare_shape_f32(int D, int id) { return shapes_of<float>(D).configure(id); }
size_t sweep_smem_f32(int D, int id) { return shapes_of<float>(D).smem(id); }
int tile_mode_f32(int D, int id) { return shapes_of<float>(D).mode(id); }

cudaError_t launch_step_f32(const Geo& g, const Bufs<float>& hb, const Inst<float>* in, int cur, cudaStream_t s, cudaEvent_t* ev,
                            const void* phi_in) {
    return shapes_of<float>(g.D).step(g.tile_id, g, hb, in, cur, s, ev, phi_in);
}
bool batch_persistent_f32(int D, int id) { return shapes_of<float>(D).persistent(id); }
cudaError_t launch_batch_persist_f32(int D, int id, const PHead* h, const PItem* it, const Inst<float>* in, int* cur,
                                     PState* st, int nsteps, int wait_log2, int test_hook, cudaStream_t s) {
    return shapes_of<float>(D).persist(id, h, it, in, cur, st, nsteps, wait_log2, test_hook, s);
}
cudaError_t launch_batch_step_f32(const BatchPlan& p, const Inst<float>* insts, int* cur, cudaStream_t s) {
    return run_batch_step<float>(p, insts, cur, s);
}
cudaError_t launch_init_f32(const Geo& g, const Inst<float>* in, int cur, const double* f, cudaStream_t s) {
    return run_init<float>(g, in, cur, f, s);
}
cudaError_t launch_cellc_f32(const Geo& g, const Inst<float>* in, int cur, cudaStream_t s) {
    return run_cellc<float>(g, in, cur, s);
}
cudaError_t launch_stress_f32(const Geo& g, const Inst<float>* in, int cur, double* out, cudaStream_t s) {
    return run_stress<float>(g, in, cur, out, s);
}
cudaError_t launch_finalise_f32(const Geo& g, const Inst<float>* in, int cur, cudaStream_t s) {
    return run_finalise<float>(g, in, cur, s);
}

}  // namespace cdg
