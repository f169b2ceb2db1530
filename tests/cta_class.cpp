// The Phase-1 kernel on at most 32 classes of ranks (sinkhorn_class.cu) on a CPU.
#include "cta.h"

#include "taot_internal.cuh"
#undef TAOT_CUDA_OK
#define TAOT_CUDA_OK(call) ((void)0)           // (the launcher's calls: nothing here launches)
#include "sinkhorn_class.cu"

namespace {

ClassArgs args;
int problems;

template <int NC, int VPL, bool TOL, int PPC>
void run()
{
    args.solvers = (problems + PPC - 1) / PPC;
    cta::blocks = args.solvers;
    for (int b = 0; b < args.solvers; ++b) cta::launch(b, kThreads, [] { sinkhorn_class_kernel<NC, VPL, TOL, PPC>(args, problems); });
}
template <bool TOL, int PPC>
int run(int nc)
{
    if (nc == 2) run<2, 2, TOL, PPC>();
    else if (nc == 8) run<8, 1, TOL, PPC>();
    else return -1;
    return nc;
}

}  // namespace

// returns the number of classes the kernel is built for
extern "C" int cta_classes(int B, int R, int share, const float* s, const float* d, const float* C, const double* rowlse0, double inv_eps, int max_iters,
                           float tol, float* plan, int32_t* iters, float* row_err, int32_t* info)
{
    taot_class_plan p;
    taot_build_classes(&p, C, R);
    if (p.kind != 1) return -1;
    std::vector<double> lse0(p.slot_rep.size(), 0.0);
    for (size_t q = 0; q < lse0.size(); ++q)
        if (p.slot_rep[q] >= 0) lse0[q] = rowlse0[p.slot_rep[q]];
    args = ClassArgs();
    SinkArgs& a = args.a;
    a.s = s; a.d = d; a.C = C; a.rowlse0 = rowlse0; a.plan = plan; a.iters = iters; a.row_err = row_err; a.info = info;
    a.R = R; a.inv_eps = inv_eps; a.eps0 = 1e-8f; a.max_iters = max_iters; a.tol = tol; a.check_every = 1;
    args.cls = p.cls.data(); args.off = p.off.data(); args.list = p.list.data(); args.lse0 = lse0.data(); args.cost = p.cost.data();
    args.cluster = 1;
    problems = B;
    if (tol > 0.0f) return share ? run<true, 4>(p.nc) : run<true, 1>(p.nc);
    return share ? run<false, 4>(p.nc) : run<false, 1>(p.nc);
}
