// The Phase-1 kernel of batches of at most 32 ranks (sinkhorn_tile.cuh, a warp per problem) on a CPU.
#include "cta.h"

#include "sinkhorn_tile.cuh"

namespace {

SinkArgs args;

template <bool TOL>
void run(int B)
{
    for (int b = 0; b < B; ++b) cta::launch(b, 32, [] { sinkhorn_tile_kernel<1, 1, 4, 8, 16, 32, TOL>(args, INT64_MAX); });
}

}  // namespace

extern "C" void cta_sinkhorn(int B, int R, const float* s, const float* d, const float* C, const double* rowlse0, double inv_eps, int max_iters,
                             float tol, int check_every, float* plan, int32_t* iters, float* row_err, int32_t* info)
{
    args = SinkArgs();
    args.s = s; args.d = d; args.C = C; args.rowlse0 = rowlse0; args.plan = plan; args.iters = iters; args.row_err = row_err; args.info = info;
    args.R = R; args.inv_eps = inv_eps; args.eps0 = 1e-8f; args.max_iters = max_iters; args.tol = tol; args.check_every = check_every;
    if (tol > 0.0f) run<true>(B);
    else run<false>(B);
}
