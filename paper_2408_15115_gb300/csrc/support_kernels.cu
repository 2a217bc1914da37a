// support_kernels.cu -- the single-run launches of the support-box moments
// (u*, sigma of Eq. 10 at t + 1) and of the marker binning (block code in
// support_moments.cuh).  Two launches: the lists depend on the markers alone
// and are built beside the near region's collide+stream.
#include "support_moments.cuh"

namespace turret {

template <int ST>
__global__ void __launch_bounds__(MB_THREADS) k_box_moments(Geom g, const typename Codec<ST>::T *__restrict__ src,
                                                            const float *__restrict__ utop_in,
                                                            const DevState *__restrict__ st, int slot, BoxGeom box,
                                                            BoxArrays ba, float rmin, float rmax) {
    pdl_trigger();
    moments_block<ST>(g, src, utop_in, st, slot, box, ba, rmin, rmax, blockIdx.x);
}

__global__ void __launch_bounds__(MB_THREADS) k_bin(DevState *st, int slot, BoxGeom box, int nm, MarkerArrays m, int cap,
                                                    float rmin, float rmax) {
    pdl_trigger();
    pdl_wait();
    bin_block(st, slot, box, nm, m.base, m.seg, m.tile_list, m.tile_count, cap, st, rmin, rmax, blockIdx.x);
}

__global__ void __launch_bounds__(QUIET_THREADS, 16) k_bin_quiet(DevState *st, int slot, BoxGeom box, int nm,
                                                                 MarkerArrays m, int cap, float rmin, float rmax) {
    constexpr int W = QUIET_THREADS / 32;
    for (int t = blockIdx.x * W + (threadIdx.x >> 5); t < box.tx * box.ty * box.tz; t += gridDim.x * W)
        bin_warp(st, slot, box, nm, m, cap, st, rmin, rmax, t, threadIdx.x & 31);
}

cudaError_t launch_box_moments(const Geom &g, int storage, const void *src, const float *utop_in, const DevState *st,
                               int slot, const BoxGeom &box, BoxArrays ba, float rmin, float rmax, cudaStream_t s) {
    const unsigned nb = (unsigned)((box.nbox + MB_THREADS - 1) / MB_THREADS);
    switch (storage) {
        case ST_F32: k_box_moments<ST_F32><<<nb, MB_THREADS, 0, s>>>(g, (const float *)src, utop_in, st, slot, box, ba, rmin, rmax); break;
        case ST_F16: k_box_moments<ST_F16><<<nb, MB_THREADS, 0, s>>>(g, (const __half *)src, utop_in, st, slot, box, ba, rmin, rmax); break;
        default: k_box_moments<ST_BF16><<<nb, MB_THREADS, 0, s>>>(g, (const __nv_bfloat16 *)src, utop_in, st, slot, box, ba, rmin, rmax); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_bin(DevState *st, int slot, const BoxGeom &box, int nm, const MarkerArrays &m, int cap, float rmin,
                       float rmax, int mode, cudaStream_t s) {
    if (mode == LISTS_QUIET) {
        k_bin_quiet<<<QUIET_BLOCKS, QUIET_THREADS, 0, s>>>(st, slot, box, nm, m, cap, rmin, rmax);
        return cudaGetLastError();
    }
    const unsigned nb = (unsigned)(box.tx * box.ty * box.tz);
    if (mode == LISTS_OVERLAP) return launch_pdl(k_bin, nb, MB_THREADS, s, st, slot, box, nm, m, cap, rmin, rmax);
    k_bin<<<nb, MB_THREADS, 0, s>>>(st, slot, box, nm, m, cap, rmin, rmax);
    return cudaGetLastError();
}

}  // namespace turret
