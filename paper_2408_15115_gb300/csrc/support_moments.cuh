// support_moments.cuh -- block code of the support-box moments and of the
// marker binning that feeds the immersed-boundary transfers (two launches on
// two streams, single runs and batches alike); the pull and moment code is the
// collide+stream's (lbm_cell.cuh), so both see identical populations.
#pragma once
#include "lbm_cell.cuh"

namespace turret {

constexpr int MB_THREADS = 128;

// Tile lists.  For one TILE^3 tile of the support box, two lists in marker
// order (ordered compaction with warp ballots; no atomics): list 0, the
// markers whose 4x4x4 stencil overlaps the tile (spreading); list 1, those
// whose stencil overlaps the stencil of any marker based in the tile (rows of
// A).  Reads the markers and the window slot only, with ordinary loads: a
// launch may start beside the particle update that writes them (pdl_wait), and
// read-only loads could be moved ahead of that wait.
// Two forms.  bin_block, a block per tile: the shortest latency, for a single
// run, whose rows of A wait for it (93x70x151, 24 steps: 1366 us; 1421 us with
// a warp per tile).
__device__ __forceinline__ void bin_block(const DevState *st, int slot, const BoxGeom &box, int nm,
                                          const int *mbase, const int *mseg,
                                          int *tile_list, int *tile_count, int cap,
                                          DevState *stw, float rmin, float rmax, int tile) {
    constexpr int NW = MB_THREADS / 32;
    const int tx = tile % box.tx, ty = (tile / box.tx) % box.ty, tz = tile / (box.tx * box.ty);
    const int t0[3] = {TILE * tx, TILE * ty, TILE * tz};
    {
        // Both lists hold markers whose stencil base b lies in [t0 - 3, t0 + 6]
        // per axis, i.e. whose position X lies in [t0 - 2, t0 + 8).  Markers
        // sit at rmin <= |X - C| <= rmax (body-frame radii, up to rounding):
        // a region outside that shell has no candidates.
        const BodySlot &S = st->s[slot];
        float dmin2 = 0.0f, dmax2 = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float c = (float)(S.Ci[a] - S.box_lo[a]) + (float)S.Cf[a];
            const float lo = (float)(t0[a] - 2), hi = (float)(t0[a] + 8);
            const float dn = fmaxf(fmaxf(lo - c, c - hi), 0.0f);
            const float dx = fmaxf(fabsf(c - lo), fabsf(c - hi));
            dmin2 += dn * dn;
            dmax2 += dx * dx;
        }
        const float margin = 0.25f;
        if (dmin2 > (rmax + margin) * (rmax + margin) ||
            (rmin > margin && dmax2 < (rmin - margin) * (rmin - margin))) {
            if (threadIdx.x < 2) tile_count[threadIdx.x * (box.tx * box.ty * box.tz) + tile] = 0;
            return;
        }
    }
    // CU chunks of MB_THREADS markers per pass: their loads are issued
    // together and their hits compacted chunk after chunk (marker order);
    // one barrier per pass, the warp counts alternating between two buffers
    constexpr int CU = 4;
    __shared__ int wcount[2][CU][2][NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nseg = (nm + MARKER_SEG - 1) / MARKER_SEG;
    int tot[2] = {0, 0};  // identical in every thread
    int par = 0;
    for (int group = 0; group < nm; group += CU * MB_THREADS) {
        // skip chunks whose segments' stencil bases all miss [t0 - 3, t0 + 6];
        // the test is the same in every thread, so a group with no chunk
        // left is skipped whole, barrier included
        bool reach[CU], any = false;
#pragma unroll
        for (int u = 0; u < CU; ++u) {
            const int chunk = group + u * MB_THREADS;
            reach[u] = false;
            for (int sg = chunk / MARKER_SEG; sg < nseg && sg * MARKER_SEG < chunk + MB_THREADS; ++sg) {
                const int *bb = mseg + 6 * sg;
                bool in = true;
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    in = in && bb[3 + a] + 3 >= t0[a] && bb[a] <= t0[a] + TILE + 2;
                reach[u] = reach[u] || in;
            }
            any = any || reach[u];
        }
        if (!any) continue;
        int pb[CU];
#pragma unroll
        for (int u = 0; u < CU; ++u) {
            const int k = group + u * MB_THREADS + tid;
            pb[u] = (reach[u] && k < nm) ? mbase[k] : -1;  // culled chunks load nothing
        }
        unsigned bal[CU][2];
        bool hit[CU][2];
#pragma unroll
        for (int u = 0; u < CU; ++u) {
            hit[u][0] = hit[u][1] = pb[u] >= 0;
            const int b[3] = {pb[u] & 1023, (pb[u] >> 10) & 1023, (pb[u] >> 20) & 1023};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const bool lo = b[a] + 3 >= t0[a];
                hit[u][0] = hit[u][0] && lo && (b[a] <= t0[a] + TILE - 1);  // stencil overlaps the tile
                hit[u][1] = hit[u][1] && lo && (b[a] <= t0[a] + TILE + 2);  // ... or a stencil based in it
            }
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                bal[u][l] = __ballot_sync(0xffffffffu, hit[u][l]);
                if (lane == 0) wcount[par][u][l][warp] = __popc(bal[u][l]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < CU; ++u)
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                int off = tot[l], sum = 0;
                for (int w = 0; w < NW; ++w) {
                    const int c = wcount[par][u][l][w];
                    off += (w < warp) ? c : 0;
                    sum += c;
                }
                if (hit[u][l]) {
                    const int pos = off + __popc(bal[u][l] & ((1u << lane) - 1u));
                    if (pos < cap)
                        tile_list[((size_t)l * (box.tx * box.ty * box.tz) + tile) * cap + pos] =
                            group + u * MB_THREADS + tid;
                }
                tot[l] += sum;
            }
        par ^= 1;
    }
    if (tid < 2) {
        tile_count[tid * (box.tx * box.ty * box.tz) + tile] = tot[tid] < cap ? tot[tid] : cap;
        if (tot[tid] > cap) atomicCAS(&stw->status, 0, STAT_OVERFLOW);
    }
}

// bin_warp, a warp per tile, for batches and for lists built well ahead of their
// use: its lanes test 32 marker segments at
// once (the bounding boxes of their stencil bases), then the markers of the
// segments that reach the tile go by in fours of 32.  Most tiles of a box reach
// few segments or none, so a tile costs a block's start, not work; four tiles
// share one.  (Moments and lists of 32 runs, 18,444 tiles: 124 us in one launch
// with a block per tile; now 38 and 31 us.)
constexpr int BIN_TILES = MB_THREADS / 32;

__device__ __forceinline__ void bin_warp(const DevState *st, int slot, const BoxGeom &box, int nm, const MarkerArrays &m,
                                         int cap, DevState *stw, float rmin, float rmax, int tile, int lane) {
    const int ntiles = box.tx * box.ty * box.tz;
    if (tile >= ntiles) return;
    const int tx = tile % box.tx, ty = (tile / box.tx) % box.ty, tz = tile / (box.tx * box.ty);
    const int t0[3] = {TILE * tx, TILE * ty, TILE * tz};
    int *count = m.tile_count + tile;
    {
        // Both lists hold markers whose stencil base b lies in [t0 - 3, t0 + 6]
        // per axis, i.e. whose position X lies in [t0 - 2, t0 + 8).  Markers
        // sit at rmin <= |X - C| <= rmax (body-frame radii, up to rounding):
        // a region outside that shell has no candidates.
        const BodySlot &S = st->s[slot];
        float dmin2 = 0.0f, dmax2 = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float c = (float)(S.Ci[a] - S.box_lo[a]) + (float)S.Cf[a];
            const float lo = (float)(t0[a] - 2), hi = (float)(t0[a] + 8);
            const float dn = fmaxf(fmaxf(lo - c, c - hi), 0.0f);
            const float dx = fmaxf(fabsf(c - lo), fabsf(c - hi));
            dmin2 += dn * dn;
            dmax2 += dx * dx;
        }
        const float margin = 0.25f;
        if (dmin2 > (rmax + margin) * (rmax + margin) ||
            (rmin > margin && dmax2 < (rmin - margin) * (rmin - margin))) {
            if (lane < 2) count[lane * ntiles] = 0;
            return;
        }
    }
    constexpr int CU = MARKER_SEG / 32;
    const int nseg = (nm + MARKER_SEG - 1) / MARKER_SEG;
    int *list = m.tile_list + (size_t)tile * cap;
    int tot[2] = {0, 0};  // identical in every lane
    for (int s0 = 0; s0 < nseg; s0 += 32) {
        bool reach = s0 + lane < nseg;
        if (reach) {
            const int *bb = m.seg + 6 * (s0 + lane);
#pragma unroll
            for (int a = 0; a < 3; ++a) reach = reach && bb[3 + a] + 3 >= t0[a] && bb[a] <= t0[a] + TILE + 2;
        }
        unsigned todo = __ballot_sync(0xffffffffu, reach);
        int pb[CU];
        auto fetch = [&](int sg) {
#pragma unroll
            for (int u = 0; u < CU; ++u) {
                const int k = sg * MARKER_SEG + u * 32 + lane;
                pb[u] = k < nm ? m.base[k] : -1;
            }
        };
        if (todo) fetch(s0 + __ffs(todo) - 1);
        while (todo) {
            const int sg = s0 + __ffs(todo) - 1;
            todo &= todo - 1;
            int cur[CU];
#pragma unroll
            for (int u = 0; u < CU; ++u) cur[u] = pb[u];
            if (todo) fetch(s0 + __ffs(todo) - 1);  // the next segment's markers, beside this one's
#pragma unroll
            for (int u = 0; u < CU; ++u) {
                const int b[3] = {cur[u] & 1023, (cur[u] >> 10) & 1023, (cur[u] >> 20) & 1023};
                bool hit[2];
                hit[0] = hit[1] = cur[u] >= 0;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const bool lo = b[a] + 3 >= t0[a];
                    hit[0] = hit[0] && lo && (b[a] <= t0[a] + TILE - 1);  // stencil overlaps the tile
                    hit[1] = hit[1] && lo && (b[a] <= t0[a] + TILE + 2);  // ... or a stencil based in it
                }
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const unsigned bal = __ballot_sync(0xffffffffu, hit[l]);
                    if (hit[l]) {
                        const int pos = tot[l] + __popc(bal & ((1u << lane) - 1u));
                        if (pos < cap) list[(size_t)l * ntiles * cap + pos] = sg * MARKER_SEG + u * 32 + lane;
                    }
                    tot[l] += __popc(bal);
                }
            }
        }
    }
    if (lane < 2) {
        const int t = lane ? tot[1] : tot[0];
        count[lane * ntiles] = t < cap ? t : cap;
        if (t > cap) atomicCAS(&stw->status, 0, STAT_OVERFLOW);
    }
}

// K2: u* and the stress of Eq. 10, sigma = -p I + (1/(2 tau) - 1) P1 with p =
// c_s^2 (rho - 1), at every support-box cell, from f(t+1) pulled from the
// post-collision buffer (box cells outside a closed face get zeros; cells no
// stencil reads, the outer layer among them, are skipped).
template <int ST>
__device__ __forceinline__ void moments_block(const Geom &g, const typename Codec<ST>::T *__restrict__ src,
                                              const float *__restrict__ utop_in, const DevState *__restrict__ st,
                                              int slot, const BoxGeom &box, const BoxArrays &ba, float rmin, float rmax,
                                              int blk) {
    const long long b = (long long)blk * blockDim.x + threadIdx.x;
    if (b >= box.nbox) return;
    const int bx = (int)(b % box.Bx);
    const int by = (int)((b / box.Bx) % box.By);
    const int bz = (int)(b / ((long long)box.Bx * box.By));
    // The outermost layer of the box is never read: along each axis a stencil
    // of a point P with |P_a - C_a| <= R = rmax + F_OFFSET covers cells
    // floor(C_a - R) - 1 .. floor(C_a + R) + 2, inside the box's
    // Ci - rc - 1 .. Ci + rc + 2 (rc = ceil R).  Skipping it keeps every pull
    // of this kernel inside the box, which is the near region: the moments
    // then depend on the near launch only, never on the far one.
    if (bx == 0 || by == 0 || bz == 0 || bx == box.Bx - 1 || by == box.By - 1 || bz == box.Bz - 1) return;
    {
        // The moments are read only inside the 4x4x4 stencils of the markers
        // (u*) and of the offset points X + F_OFFSET n (sigma, p).  Those points
        // lie at rmin - F_OFFSET <= |P - C| <= rmax + F_OFFSET, and a stencil
        // cell within 2 cells of P per axis (2 sqrt 3 in all): cells outside
        // that shell (the corners of the box, the core of a large body) are
        // never read and are skipped.
        const BodySlot &S = st->s[slot];
        const int bb[3] = {bx, by, bz};
        float d2 = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float d = (float)bb[a] - ((float)(S.Ci[a] - S.box_lo[a]) + (float)S.Cf[a]);
            d2 += d * d;
        }
        const float reach = F_OFFSET + 3.4641016f + 0.25f;
        if (d2 > (rmax + reach) * (rmax + reach) || (rmin > reach && d2 < (rmin - reach) * (rmin - reach))) return;
    }
    int c[3] = {st->s[slot].box_lo[0] + bx, st->s[slot].box_lo[1] + by, st->s[slot].box_lo[2] + bz};
    const int n[3] = {g.nx, g.ny, g.nz};
    const bool per[3] = {g.bc_x == BC_PERIODIC, g.bc_y == BC_PERIODIC, g.bc_bottom == BC_PERIODIC};
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (per[a]) {
            c[a] %= n[a];
            if (c[a] < 0) c[a] += n[a];
        } else if (c[a] < 0 || c[a] >= n[a]) {
            inside = false;
        }
    }
    if (!inside) {
        ba.u[b] = ba.s[2 * b] = ba.s[2 * b + 1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        return;
    }
    float q[27];
    pull27<ST>(g, src, c[0], c[1], c[2], st->s[slot].ring, st->s[slot].reseed, utop_in, q);
    const MacroR<float> M = macro_raw<ST>(moments_raw<ST>(q));
    const float tau = tau_of(g, c[2]);
    // (1/(2 tau) - 1) P1 with P1 = P1~ / 216 = P / (216 K)
    const float k2 = (0.5f / tau - 1.0f) * (INV_SCALE / Codec<ST>::K);
    const float p = M.drho * (1.0f / 3.0f);
    ba.u[b] = make_float4(M.ux, M.uy, M.uz, 0.0f);
    ba.s[2 * b] = make_float4(-p + k2 * M.Pxx, -p + k2 * M.Pyy, -p + k2 * M.Pzz, k2 * M.Pxy);
    ba.s[2 * b + 1] = make_float4(k2 * M.Pxz, k2 * M.Pyz, p, 0.0f);
}

}  // namespace turret
