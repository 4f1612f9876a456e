// gp_eval_r8_f2.cu -- instances of the batched evaluator: 8 rows per
// thread, feature mode 2 (columns 0 and 1 held in registers),
// program classes 0 (6 stack slots) and 2 (7 slots, tan and the extended
// functions; the others always run 4 rows per thread), with the loss epilogue, the moment epilogue of the correlation fitness, or the
// store epilogue (predictions).
#include "gp_interp.cuh"

namespace gpk {
namespace {
template <int EPI>
cudaError_t launch_cls(const EvalArgs &a, int grid, int block, cudaStream_t st) {
    if (a.cls == kClassShallowExt)
        return launch_eval_t<8, kSmallDepth - 1, 2, EPI, true>(a, grid, block, st);
    return launch_eval_t<8, kShallowDepth - 1, 2, EPI, false>(a, grid, block, st);
}
template <int EPI>
int info_cls(int cls, int block, int *regs) {
    if (cls == kClassShallowExt) return info_t<8, kSmallDepth - 1, 2, EPI, true>(block, regs);
    return info_t<8, kShallowDepth - 1, 2, EPI, false>(block, regs);
}
}  // namespace

cudaError_t launch_eval_r8_f2(const EvalArgs &a, int grid, int block, cudaStream_t st) {
    if (a.cls != kClassShallow && a.cls != kClassShallowExt) return cudaErrorInvalidValue;
    if (a.pred) return launch_cls<kEpiPred>(a, grid, block, st);
    return a.mom ? launch_cls<kEpiMom>(a, grid, block, st) : launch_cls<kEpiLoss>(a, grid, block, st);
}
int info_eval_r8_f2(int cls, int block, int *regs, bool moments, bool pred) {
    if (cls != kClassShallow && cls != kClassShallowExt) return 0;
    if (pred) return info_cls<kEpiPred>(cls, block, regs);
    return moments ? info_cls<kEpiMom>(cls, block, regs) : info_cls<kEpiLoss>(cls, block, regs);
}
}  // namespace gpk
