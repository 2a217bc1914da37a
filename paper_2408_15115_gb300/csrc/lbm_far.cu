// lbm_far.cu -- the far-cell collide+stream of a coupled single-run step with
// FP32 storage, under a register cap.
//
// In the step graph this launch shares the SMs with the immersed-boundary
// chain.  At 128 registers its four resident blocks of 128 threads fill the
// 65,536-register file, so any chain block resident on an SM displaces one of
// them (a quarter of that SM's streaming).  At 120 registers (four values of the
// boundary path spilled, 16 bytes) four blocks leave 4,096 registers free, room
// for a small chain block (the 64-thread interpolation blocks) beside them.  The cell code is the same
// device function as every other collide+stream launch (lbm_cell.cuh), so
// results are identical.
#include "lbm_cell.cuh"

namespace turret {

__global__ void __maxnreg__(120) k_collide_stream_far_f32(Geom g, const float *__restrict__ src,
                                                          float *__restrict__ dst, const float *__restrict__ utop_in,
                                                          float *__restrict__ utop_out, const BodySlot *win,
                                                          const float *__restrict__ hbox, BoxGeom box, int flat) {
    int cx, cy;
    window_cell(g, flat, cx, cy);
    k1_pair<ST_F32, K1_FAR>(g, src, dst, utop_in, utop_out, *win, hbox, box, cx, cy, 2 * blockIdx.z);
}

cudaError_t launch_collide_far(const Geom &g, int storage, const void *src, void *dst, const float *utop_in,
                               float *utop_out, DevState *st, const BodySlot *win, const float *hbox, const BoxGeom &box,
                               cudaStream_t s, const CUtensorMap *lmap, const CUtensorMap *smap) {
    if (storage != ST_F32 && lmap && smap)
        return launch_collide_staged(g, storage, *lmap, *smap, src, dst, utop_in, utop_out, st, win, -1, hbox, box,
                                     REGION_FAR, s);
    if (storage != ST_F32 && xpair_eligible(g, storage))
        return launch_collide_xpair(g, storage, src, dst, utop_in, utop_out, st, win, -1, hbox, box, REGION_FAR, s);
    if (storage != ST_F32)
        return launch_collide_stream(g, storage, src, dst, utop_in, utop_out, st, win, -1, hbox, box, true,
                                     REGION_FAR, s);
    k_collide_stream_far_f32<<<window_grid(g, ST_F32, (g.nz + 1) / 2), dim3(32, 4), 0, s>>>(  // one thread per pair of planes
        g, (const float *)src, (float *)dst, utop_in, utop_out, win, hbox, box, window_flat(g, ST_F32));
    return cudaGetLastError();
}

bool is_far_kernel(const void *fn) { return fn == (const void *)k_collide_stream_far_f32; }

}  // namespace turret
