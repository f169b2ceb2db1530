// The Phase-1 kernel of few problems (sinkhorn_split.cuh) on a CPU.
#include "cta.h"

#include "sinkhorn_split.cuh"

namespace {

SinkArgs args;

template <int RMAX, int NT>
void run(int B)
{
    for (int b = 0; b < B; ++b) {
        if (args.tol > 0.0f) cta::launch(b, NT, [] { sinkhorn_tile_kernel<RMAX, NT, true>(args); });
        else cta::launch(b, NT, [] { sinkhorn_tile_kernel<RMAX, NT, false>(args); });
    }
}

// neighbours exchange a word, with and without a wait
uint32_t box[64];
template <int ORDERS>
void exchange()
{
    box[cta::me] = cta::me;
    if (ORDERS) __syncthreads();
    else if (__any_sync(~0u, cta::me < 0)) return;
    box[(cta::me + 1) % 32 + cta::me / 32 * 32] += 1;
}

}  // namespace

extern "C" {

void cta_exchange(int orders) { cta::launch(0, 64, orders ? exchange<1> : exchange<0>); }

void cta_sinkhorn(int B, int R, int threads, const float* s, const float* d, const float* C, const double* rowlse0, double inv_eps, int max_iters,
                  float tol, int check_every, float* plan, int32_t* iters, float* row_err, int32_t* info)
{
    args = SinkArgs();
    args.s = s; args.d = d; args.C = C; args.rowlse0 = rowlse0; args.plan = plan; args.iters = iters; args.row_err = row_err; args.info = info;
    args.R = R; args.inv_eps = inv_eps; args.eps0 = 1e-8f; args.max_iters = max_iters; args.tol = tol; args.check_every = check_every;
    if (R <= 32) run<32, 128>(B);
    else if (threads == 128) run<64, 128>(B);
    else run<64, 64>(B);
}

}
