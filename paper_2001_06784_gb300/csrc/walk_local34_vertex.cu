// Per-vertex counts with bitsets of 3 and 4 words.
#include "local.cuh"

namespace pvt {

template pvt_status launch_local<3, MODE_VERTEX>(pvt_dag *, const CountArgs &, int, cudaStream_t);
template pvt_status launch_local<4, MODE_VERTEX>(pvt_dag *, const CountArgs &, int, cudaStream_t);
template pvt_status launch_local_batch<4, MODE_VERTEX>(const BatchGraph *, const uint64_t *, unsigned, unsigned *,
                                                     const unsigned long long *, int, unsigned *,
                                                     unsigned long long *, int, size_t, cudaStream_t);

}  // namespace pvt
