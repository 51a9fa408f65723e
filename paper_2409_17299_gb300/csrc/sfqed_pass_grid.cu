// Pass kernels for the gridded field (trilinear interpolation of the
// caller's node values, one PIC step's fields).
#define SFQ_GRID 1
#define SFQ_PASS_NS pass_grid
#include "sfqed_pass.cuh"

template qed_status sfq::pass_grid::launch_pass<float>(qed_ctx *, sfq::PassArgs &, bool,
    cudaGraphConditionalHandle, int);
template qed_status sfq::pass_grid::launch_pass<double>(qed_ctx *, sfq::PassArgs &, bool,
    cudaGraphConditionalHandle, int);
template qed_status sfq::pass_grid::launch_od<float>(qed_ctx *, sfq::PassArgs &, bool);
template qed_status sfq::pass_grid::launch_od<double>(qed_ctx *, sfq::PassArgs &, bool);
template qed_status sfq::pass_grid::launch_steps<float>(qed_ctx *, sfq::PassArgs &, int64_t, int, int);
template int sfq::pass_grid::steps_blocks<float>(const qed_ctx *, int64_t, int);
template qed_status sfq::pass_grid::launch_steps<double>(qed_ctx *, sfq::PassArgs &, int64_t, int, int);
template int sfq::pass_grid::steps_blocks<double>(const qed_ctx *, int64_t, int);
