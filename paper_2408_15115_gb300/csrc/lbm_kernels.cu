// lbm_kernels.cu -- single-run kernels of the fused collide+stream and of the
// passes sharing its streaming and moment code (cell code in lbm_cell.cuh).
#include "lbm_cell.cuh"

namespace turret {

// The near region as one flat range of cells, x fastest: every thread but those
// of the last block has a cell (rows of 26 to 46 cells leave 19 to 28 % of the
// lanes of 32-wide rows idle, and the launch of a large body a second, nearly
// empty wave: 46^3 cells 1152 blocks on 912 places, 761 flat; 864 where a body
// needs a layer around the box, 256x256x512 18,958 -> 19,037 us per 16 steps,
// 32x32x64 4190 -> 4249 per 100: the reason for NEAR_SLACK).
template <int ST>
__device__ __forceinline__ void near_cell(const Geom &g, const typename Codec<ST>::T *__restrict__ src,
                                          typename Codec<ST>::T *__restrict__ dst, const float *__restrict__ utop_in,
                                          float *__restrict__ utop_out, const BodySlot &S,
                                          const float *__restrict__ hbox, const BoxGeom &box) {
    const int ex = box.Nx, ey = box.Ny, ez = box.Nz;
    const int i = blockIdx.x * 128 + threadIdx.y * 32 + threadIdx.x;
    if (i < ex * ey * ez)
        k1_cell<ST, K1_NEAR>(g, src, dst, utop_in, utop_out, S, hbox, box, i % ex, (i / ex) % ey, i / (ex * ey));
}

// Window launches with 16-bit storage: five blocks per SM (96 registers; 88 to
// 104 bytes of spills in L1, 456 loaded with forcing) measured faster than four;
// FP32 keeps four (128 registers; 28 bytes with forcing); the small near-region
// launch is left unconstrained.  The spills are those of the boundary path
// (pull27_edge), which pays wherever a window has closed faces (130x131x160
// between walls FP16 256 -> 134 us) and costs where it has none at most 1.6 %
// (160^3 periodic FP16 94.6 -> 96.1; BF16 96.4 -> 95.4, FP32 134.9 -> 134.7).
template <int ST, int MODE>
__global__ void __launch_bounds__(128, MODE == K1_NEAR ? 1 : (ST == ST_F32 ? 4 : 5)) k_collide_stream(Geom g, const typename Codec<ST>::T *__restrict__ src,
                                                        typename Codec<ST>::T *__restrict__ dst,
                                                        const float *__restrict__ utop_in,
                                                        float *__restrict__ utop_out, DevState *st,
                                                        const BodySlot *win, int slot_out, const float *__restrict__ hbox, BoxGeom box,
                                                        int flat) {
    if (slot_out >= 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0 &&
        threadIdx.y == 0) {
        // carry the body and window to the next time level (no entering plane there)
        st->s[slot_out] = *win;
        st->s[slot_out].reseed = -1;
        st->s[slot_out].step += 1;
    }
    if constexpr (MODE == K1_NEAR) {  // small, on the critical path: one cell per thread
        near_cell<ST>(g, src, dst, utop_in, utop_out, *win, hbox, box);
    } else {  // the window: a pair of planes per thread
        int cx, cy;
        window_cell(g, flat, cx, cy);
        k1_pair<ST, MODE>(g, src, dst, utop_in, utop_out, *win, hbox, box, cx, cy, 2 * blockIdx.z);
    }
}


// Equilibrium of given (rho - 1, u) fields (doubles, window order) as the
// post-collision state; u of the top plane goes to the pressure-ghost buffer.
template <int ST>
__global__ void k_init_equilibrium(Geom g, typename Codec<ST>::T *__restrict__ dst, const double *__restrict__ drho,
                                   const double *__restrict__ u, float *__restrict__ utop) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.ncell) return;
    MacroR<float> M;
    M.drho = drho ? (float)drho[c] : 0.0f;
    M.rho = (float)(1.0 + (drho ? drho[c] : 0.0));
    M.ux = u ? (float)u[3 * c] : 0.0f;
    M.uy = u ? (float)u[3 * c + 1] : 0.0f;
    M.uz = u ? (float)u[3 * c + 2] : 0.0f;
    M.Pxx = M.Pyy = M.Pzz = M.Pxy = M.Pxz = M.Pyz = 0.0f;
    float q[27];
    const float h[3] = {0.0f, 0.0f, 0.0f};
    collide_rr<ST>(M, 1.0f, false, 1.0f, 0.0f, 1.0f, h, q);
#pragma unroll
    for (int i = 0; i < 27; ++i) Codec<ST>::store(dst + (size_t)i * g.ncell + c, q[i]);
    const long long z = c / g.plane;
    if (z == g.nz - 1) {
        const long long p = c - z * g.plane;
        utop[p] = M.ux;
        utop[g.plane + p] = M.uy;
        utop[2 * g.plane + p] = M.uz;
    }
}

// rho, u (or the 27 pre-collision deviations) of f(t) at every cell.
template <int ST>
__global__ void __launch_bounds__(128) k_macro(Geom g, const typename Codec<ST>::T *__restrict__ src,
                                               const float *__restrict__ utop_in, const DevState *__restrict__ st,
                                               int slot, float *__restrict__ out, int pops, int flat) {
    int x, y;
    window_cell(g, flat, x, y);
    const int zl = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    float q[27];
    pull27<ST>(g, src, x, y, zl, st->s[slot].ring, st->s[slot].reseed, utop_in, q);
    const size_t c = ((size_t)zl * g.ny + y) * g.nx + x;
    if (pops) {  // f_i - w_i = s_i / 216 = r_i W_i / (216 K)
#pragma unroll
        for (int i = 0; i < 27; ++i)
            out[(size_t)i * g.ncell + c] = q[i] * ((Codec<ST>::scaled ? Wq(i) / Codec<ST>::K : 1.0f) * INV_SCALE);
        return;
    }
    const MacroR<float> M = macro_raw<ST>(moments_raw<ST>(q));
    out[c] = M.rho;
    out[g.ncell + c] = M.ux;
    out[2 * g.ncell + c] = M.uy;
    out[3 * g.ncell + c] = M.uz;
}


// ---------------------------------------------------------------------------
// Launchers.
static dim3 near_grid(const BoxGeom &b) {
    return dim3((unsigned)(((long long)b.Nx * b.Ny * b.Nz + 127) / 128));
}

template <int ST>
static cudaError_t collide_t(const Geom &g, const void *src, void *dst, const float *utop_in, float *utop_out,
                             DevState *st, const BodySlot *win, int slot_out, const float *hbox, const BoxGeom &box,
                             bool has_box, int region, cudaStream_t s, bool after_spread) {
    using T = typename Codec<ST>::T;
    const dim3 blk(32, 4);
    const T *fs = (const T *)src;
    T *fd = (T *)dst;
    if (region == REGION_NEAR && after_spread)
        return launch_pdl(k_collide_stream<ST, K1_NEAR>, near_grid(box), blk, s, g, fs, fd, utop_in, utop_out, st, win,
                          slot_out, hbox, box, 0);
    if (region == REGION_NEAR)
        k_collide_stream<ST, K1_NEAR><<<near_grid(box), blk, 0, s>>>(g, fs, fd, utop_in, utop_out, st, win, slot_out, hbox, box, window_flat(g, ST));
    else if (region == REGION_FAR)
        k_collide_stream<ST, K1_FAR><<<window_grid(g, ST, (g.nz + 1) / 2), blk, 0, s>>>(g, fs, fd, utop_in, utop_out, st, win, slot_out, hbox, box, window_flat(g, ST));
    else if (has_box)
        k_collide_stream<ST, K1_ALLF><<<window_grid(g, ST, (g.nz + 1) / 2), blk, 0, s>>>(g, fs, fd, utop_in, utop_out, st, win, slot_out, hbox, box, window_flat(g, ST));
    else
        k_collide_stream<ST, K1_ALL><<<window_grid(g, ST, (g.nz + 1) / 2), blk, 0, s>>>(g, fs, fd, utop_in, utop_out, st, win, slot_out, hbox, box, window_flat(g, ST));
    return cudaGetLastError();
}

cudaError_t launch_collide_stream(const Geom &g, int storage, const void *src, void *dst, const float *utop_in,
                                  float *utop_out, DevState *st, const BodySlot *win, int slot_out, const float *hbox,
                                  const BoxGeom &box, bool has_box, int region, cudaStream_t s, bool after_spread) {
    switch (storage) {
        case ST_F32: return collide_t<ST_F32>(g, src, dst, utop_in, utop_out, st, win, slot_out, hbox, box, has_box, region, s, after_spread);
        case ST_F16: return collide_t<ST_F16>(g, src, dst, utop_in, utop_out, st, win, slot_out, hbox, box, has_box, region, s, after_spread);
        default: return collide_t<ST_BF16>(g, src, dst, utop_in, utop_out, st, win, slot_out, hbox, box, has_box, region, s, after_spread);
    }
}

bool is_window_kernel(const void *fn) {
    return fn == (const void *)k_collide_stream<ST_F32, K1_ALL> || fn == (const void *)k_collide_stream<ST_F32, K1_ALLF> ||
           fn == (const void *)k_collide_stream<ST_F32, K1_FAR> || fn == (const void *)k_collide_stream<ST_F16, K1_ALL> ||
           fn == (const void *)k_collide_stream<ST_F16, K1_ALLF> || fn == (const void *)k_collide_stream<ST_F16, K1_FAR> ||
           fn == (const void *)k_collide_stream<ST_BF16, K1_ALL> || fn == (const void *)k_collide_stream<ST_BF16, K1_ALLF> ||
           fn == (const void *)k_collide_stream<ST_BF16, K1_FAR>;
}

cudaError_t launch_init_equilibrium(const Geom &g, int storage, void *dst, const double *drho, const double *u,
                                    float *utop, cudaStream_t s) {
    const unsigned nb = (unsigned)((g.ncell + 255) / 256);
    switch (storage) {
        case ST_F32: k_init_equilibrium<ST_F32><<<nb, 256, 0, s>>>(g, (float *)dst, drho, u, utop); break;
        case ST_F16: k_init_equilibrium<ST_F16><<<nb, 256, 0, s>>>(g, (__half *)dst, drho, u, utop); break;
        default: k_init_equilibrium<ST_BF16><<<nb, 256, 0, s>>>(g, (__nv_bfloat16 *)dst, drho, u, utop); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_macro(const Geom &g, int storage, const void *src, const float *utop_in, const DevState *st,
                         int slot, float *out, bool pops, cudaStream_t s) {
    // the caller's array is only known to hold floats: pairs are stored where it
    // is 8-byte aligned
    if (xpair_eligible(g, storage) && reinterpret_cast<uintptr_t>(out) % sizeof(float2) == 0)
        return launch_macro_xpair(g, storage, src, utop_in, st, slot, out, pops, s);
    switch (storage) {
        case ST_F32: k_macro<ST_F32><<<window_grid(g, storage, g.nz), dim3(32, 4), 0, s>>>(g, (const float *)src, utop_in, st, slot, out, pops, window_flat(g, storage)); break;
        case ST_F16: k_macro<ST_F16><<<window_grid(g, storage, g.nz), dim3(32, 4), 0, s>>>(g, (const __half *)src, utop_in, st, slot, out, pops, window_flat(g, storage)); break;
        default: k_macro<ST_BF16><<<window_grid(g, storage, g.nz), dim3(32, 4), 0, s>>>(g, (const __nv_bfloat16 *)src, utop_in, st, slot, out, pops, window_flat(g, storage)); break;
    }
    return cudaGetLastError();
}


}  // namespace turret
