// Launcher of the lane walk (lanes.cuh) over the compacted frames of the
// two-phase global count.
#include "lanes.cuh"

namespace pvt {

// Frames of a launch: those the wide walks emitted (the count capped at
// A.emit_cap; null: none) and the slots the <= 32 class's gather reserved.
__device__ __forceinline__ unsigned wide_frames(const CountArgs &A)
{
    return A.emit ? (unsigned)min(*(volatile unsigned long long *)A.emit_count, (unsigned long long)A.emit_cap) : 0u;
}
__device__ __forceinline__ unsigned all_frames(const CountArgs &A)
{
    return wide_frames(A) + (A.emit1 ? min(vload(A.emit1_count), A.emit1_cap) : 0u);
}

// Every emitted frame (A.emit, then A.emit1); walk statistics to slot
// FRAMES_SLOT, those of <= 32 class roots to their own class.
__global__ void __launch_bounds__(32 * LANE_WPB, 2) k_lanes(CountArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    LaneWork *lw = reinterpret_cast<LaneWork *>(smem);
    unsigned *sh32 = reinterpret_cast<unsigned *>(lw + LANE_WPB);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < HIST_H * HIST_P; i += blockDim.x) sh32[i] = 0;
    __syncthreads();
    lane_walk(lw[wid], sh32, A, lane, wide_frames(A), all_frames(A), NCLASS);
    hist_flush(sh32, A);
}


static pvt_status launch_lanes_kernel(pvt_dag *g, const CountArgs &A, int phase, cudaStream_t s)
{
    constexpr size_t smem = lane_smem_bytes();
    auto kern = k_lanes;
    int per_sm = 0;
    PVT_CK(resident_blocks((const void *)kern, 32 * LANE_WPB, smem, &per_sm));
    if (per_sm < 1) {
        set_error("lane walk kernel cannot be resident (shared memory)");
        return PVT_ECUDA;
    }
    const unsigned grid = (unsigned)(g->num_sms * per_sm);
    phase_begin(g, phase, s);
    kern<<<grid, 32 * LANE_WPB, smem, s>>>(A);
    PVT_CK(cudaGetLastError());
    phase_end(g, phase, s);
    return PVT_OK;
}

// Queue counters of the second phase: the frame counts are final on the device.
static __global__ void k_lanes_frames_init(CountArgs A)
{
    for (int i = threadIdx.x; i < QCTL_WORDS; i += blockDim.x) A.qctl[i] = i == Q_OUT ? all_frames(A) : 0u;
}

// Ring queue of a lane launch in the buffers of slot `q` of the dag.
static pvt_status lane_ring(pvt_dag *g, CountArgs &A, int q, cudaStream_t s)
{
    pvt_status st;
    if ((st = grow(g, g->qframes[q], (size_t)SPLIT_QCAP * FRAME_WORDS, s)) != PVT_OK) return st;
    if ((st = grow(g, g->qready[q], (size_t)SPLIT_QCAP * 2, s)) != PVT_OK || g->sizing) return st;
    PVT_CK(cudaMemsetAsync(g->qready[q].p, 0, (size_t)SPLIT_QCAP * 2 * sizeof(uint32_t), s));
    A.qframes = g->qframes[q].p;
    A.qready = g->qready[q].p;
    A.qdone = g->qready[q].p + SPLIT_QCAP;
    A.qctl = g->qctl + QCTL_WORDS * q;
    A.qcap = SPLIT_QCAP;
    return PVT_OK;
}

pvt_status launch_lanes_frames(pvt_dag *g, const CountArgs &base, cudaStream_t s)
{
    CountArgs A = base;
    A.cls = NCLASS;
    pvt_status st = lane_ring(g, A, 0, s);
    if (st != PVT_OK || g->sizing) return st;
    k_lanes_frames_init<<<1, 128, 0, s>>>(A);
    PVT_CK(cudaGetLastError());
    g->stats.launches += 2;
    return launch_lanes_kernel(g, A, PH_FRAMES, s);
}

}  // namespace pvt
