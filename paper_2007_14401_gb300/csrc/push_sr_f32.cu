// push_sr_f32.cu -- mixed path: FP32 fields, momenta and arithmetic; positions
// stored in FP64 or as FP32 pairs and advanced without loss (see push_sr.cuh).
#include "push_sr.cuh"

namespace gcb {

gcb_status GCB_FN(push_step_f32)(const gcb_particles *p, const gcb_particles *in, const gcb_grid *g,
                         const gcb_params *prm, cudaStream_t st, unsigned long long *stats,
                         int nsteps)
{
    if (p->pos_mode == GCB_POS_F32PAIR)
        return dispatch_push<float, 1>(p, in, g, prm, st, stats, nsteps);
    return dispatch_push<float, 0>(p, in, g, prm, st, stats, nsteps);
}

// One step of the adjoint's forward run (2D, gradient records), in the
// arrangement the adjoint replays (gca_step_c).  The interpolant's gradient
// jumps at cell faces, so an adjoint moves by up to 1e-3 of its rms where a
// last-place difference takes a gather point across a face: the replay has to
// see the points the forward run saw.
template <int PM>
static gcb_status step_adj(const gcb_particles *p, const gcb_particles *in, const gcb_grid *g,
                           const gcb_params *prm, cudaStream_t st, unsigned long long *stats)
{
    PushArgs<float> a;
    fill_args<float>(a, p, in, g, prm, stats);
    return launch_push<float, 2, PM, 2, false, false, false, false, true>(a, st);
}

gcb_status GCB_FN(push_step_adj_f32)(const gcb_particles *p, const gcb_particles *in, const gcb_grid *g,
                             const gcb_params *prm, cudaStream_t st, unsigned long long *stats)
{
    return p->pos_mode == GCB_POS_F32PAIR ? step_adj<1>(p, in, g, prm, st, stats)
                                          : step_adj<0>(p, in, g, prm, st, stats);
}

}  // namespace gcb
