// Pass kernels for the analytic field descriptors (uniform, rotating E,
// standing circularly polarised wave).
#define SFQ_GRID 0
#define SFQ_PASS_NS pass_analytic
#include "sfqed_pass.cuh"

template qed_status sfq::pass_analytic::launch_pass<float>(qed_ctx *, sfq::PassArgs &, bool,
    cudaGraphConditionalHandle, int);
template qed_status sfq::pass_analytic::launch_pass<double>(qed_ctx *, sfq::PassArgs &, bool,
    cudaGraphConditionalHandle, int);
template qed_status sfq::pass_analytic::launch_od<float>(qed_ctx *, sfq::PassArgs &, bool);
template qed_status sfq::pass_analytic::launch_od<double>(qed_ctx *, sfq::PassArgs &, bool);
template qed_status sfq::pass_analytic::launch_steps<float>(qed_ctx *, sfq::PassArgs &, int64_t, int, int);
template int sfq::pass_analytic::steps_blocks<float>(const qed_ctx *, int64_t, int);
template qed_status sfq::pass_analytic::launch_steps<double>(qed_ctx *, sfq::PassArgs &, int64_t, int, int);
template int sfq::pass_analytic::steps_blocks<double>(const qed_ctx *, int64_t, int);
