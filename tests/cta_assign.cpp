// The reassignment of one chunk after another (assign.cu) on a CPU, without staging.
#include "cta.h"

#include "taot_internal.cuh"
#undef TAOT_CUDA_OK
#define TAOT_CUDA_OK(call) ((void)0)           // (the launcher's calls: nothing here launches)
#include "assign.cu"

namespace {

AssignArgs args;

template <bool VEC, int NT>
void run(int blocks)
{
    for (int b = 0; b < blocks; ++b) cta::launch(b, NT, [] { assign_chunk_kernel<VEC, false, false, NT>(args); });
}

}  // namespace

extern "C" void cta_assign(int L, int R, int E, int K, long layer_elems, long seg, int nc, int vec, int threads, const int32_t* topk, const int32_t* cc,
                           const int32_t* slot_expert, const int32_t* X, int32_t* out, int32_t* info)
{
    args = AssignArgs();
    args.topk = topk; args.cc = cc; args.slot_expert = slot_expert; args.X = X; args.out = out; args.info = info;
    args.layer_elems = layer_elems; args.seg = seg; args.nc = nc; args.R = R; args.E = E; args.K = K;
    const int blocks = L * R * nc;
    if (threads == 512) vec ? run<true, 512>(blocks) : run<false, 512>(blocks);
    else vec ? run<true, 256>(blocks) : run<false, 256>(blocks);
}
