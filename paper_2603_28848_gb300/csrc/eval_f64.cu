// FP64 instantiations of the sample kernel (the parity path): with the FP32
// screen, and the plain loop for contexts whose tables leave no room for the
// screen's queues.  Two CTAs of 256 threads per SM: while one warp occupies
// its partition's FP64 pipe the others screen.
#include "eval_impl.cuh"

namespace best {
template __global__ void eval_kernel<double, 4, 2, false, 256, 2>(EvalParams);
template __global__ void eval_kernel<double, 5, 2, false, 256, 2>(EvalParams);
template __global__ void eval_kernel<double, 6, 2, false, 256, 2>(EvalParams);
template __global__ void eval_kernel<double, 4, 1>(EvalParams);
template __global__ void eval_kernel<double, 5, 1>(EvalParams);
template __global__ void eval_kernel<double, 6, 1>(EvalParams);

int eval_variants_f64(int nmax, SampleVariant* v) {
    void *fn, *fq;
    switch (nmax) {
        case 3: case 4:
            fn = reinterpret_cast<void*>(&eval_kernel<double, 4, 1>);
            fq = reinterpret_cast<void*>(&eval_kernel<double, 4, 2, false, 256, 2>);
            break;
        case 5:
            fn = reinterpret_cast<void*>(&eval_kernel<double, 5, 1>);
            fq = reinterpret_cast<void*>(&eval_kernel<double, 5, 2, false, 256, 2>);
            break;
        default:
            fn = reinterpret_cast<void*>(&eval_kernel<double, 6, 1>);
            fq = reinterpret_cast<void*>(&eval_kernel<double, 6, 2, false, 256, 2>);
            break;
    }
    v[0] = {fq, 2, 256, 2};
    v[1] = {fn, 1, 256, 1};
    return 2;
}
}  // namespace best
