// Walk kernels of global counts with bitsets of 10, 12 words, the widths between
// powers of two: a class whose largest out-degree fits one of them takes it.
#include "walk.cuh"

namespace pvt {

template pvt_status launch_class<10, MODE_GLOBAL, true>(pvt_dag *, const CountArgs &, int, cudaStream_t);
template pvt_status launch_class<12, MODE_GLOBAL, true>(pvt_dag *, const CountArgs &, int, cudaStream_t);

}  // namespace pvt
