// Detector spectra S[p, d, j] = sum_k M_d(k) I[p, j, k]  (Sec. II.B DetectorSet; App. B).
//
// Each detector is a compact list of (pixel, weight) pairs built at plan time, so only
// the pixels inside an aperture are read.  One warp per (p, d, j): lanes stride the
// list in a fixed order and combine with a fixed xor-shuffle tree, so the result does
// not depend on scheduling (deterministic).
#include "tacaw_internal.cuh"

namespace tacaw {

__global__ void aperture_kernel(ApertureArgs a) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = blockIdx.x * 8 + warp;
    const int d = blockIdx.y;
    const int p = blockIdx.z;
    if (j >= a.Nw) return;
    const float *Ipj = a.I + ((int64_t)p * a.Nw + j) * a.npix;
    float v = 0.f;
    // eight pixels in flight a lane, added in list order (one at a time the list of a 20-pixel disk, 40
    // dependent pairs of loads, took 15 us)
    const int end = a.off[d + 1];
    for (int i0 = a.off[d] + lane; i0 < end; i0 += 256) {
        float x[8], w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = i0 + 32 * k;
            w[k] = i < end ? a.wts[i] : 0.f;
            x[k] = i < end ? Ipj[a.idx[i]] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (i0 + 32 * k < end) v = fmaf(w[k], x[k], v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) a.S[((int64_t)p * a.D + d) * a.Nw + j] = v;
}

cudaError_t launch_aperture(const ApertureArgs &a, cudaStream_t st) {
    if (a.D == 0 || a.P == 0) return cudaSuccess;
    dim3 grd((a.Nw + 7) / 8, a.D, a.P);
    aperture_kernel<<<grd, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace tacaw
