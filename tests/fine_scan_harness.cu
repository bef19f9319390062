// fine_scan over weights given as tables: `sums` is what the run sums see, `single` what the look at one element sees.
#include "svip_draft.cuh"

struct TableWeights {
    const float* sums;
    const float* single;
    typedef int Raw;
    __device__ int load(int vi) const { return vi; }
    __device__ void weights(int, int vi, float (&w)[4]) const {
        for (int j = 0; j < 4; ++j) w[j] = sums[4 * vi + j];
    }
    __device__ float element(int vi, int j) const { return single[4 * vi + j]; }
};

__global__ void __launch_bounds__(svip::kThreads) scan_kernel(TableWeights wf, int v_lo, int v_hi, float target, int* out) {
    __shared__ svip::ScanShared sh;
    const int tid = threadIdx.x;
    const int r = svip::fine_scan<4>(wf, v_lo, v_hi, 0.f, target, sh, tid, tid & 31, tid >> 5);
    if (tid == 0) *out = r;
}

extern "C" int scan(const float* sums, const float* single, int v_lo, int v_hi, float target, int* out) {
    scan_kernel<<<1, svip::kThreads>>>(TableWeights{sums, single}, v_lo, v_hi, target, out);
    return static_cast<int>(cudaDeviceSynchronize());
}
