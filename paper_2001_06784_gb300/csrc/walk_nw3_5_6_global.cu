// Walk kernels of global counts with bitsets of 3, 5, 6 words, the widths between
// powers of two: a class whose largest out-degree fits one of them takes it.
#include "walk.cuh"

namespace pvt {

template pvt_status launch_class<3, MODE_GLOBAL, true>(pvt_dag *, const CountArgs &, int, cudaStream_t);
template pvt_status launch_class<5, MODE_GLOBAL, true>(pvt_dag *, const CountArgs &, int, cudaStream_t);
template pvt_status launch_class<6, MODE_GLOBAL, true>(pvt_dag *, const CountArgs &, int, cudaStream_t);

}  // namespace pvt
