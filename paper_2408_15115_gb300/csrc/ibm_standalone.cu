// ibm_standalone.cu -- the spreading operator of the immersed-boundary method
// (Sec. 2.2, step l = 1) as a standalone call on a caller grid:
//   field(x) = S[h](x) = sum_k h_k W(x - X_k) dS_k.
// The gather of the time step's spreading (4^3 tiles, candidates in marker
// order, slice sums in slice order: bitwise reproducible) on a grid that is
// mostly empty: the markers lie on a surface, so few tiles have candidates.
//
//   k_records      : every marker's stencil record, and its index appended to
//                    the lists of the 1 to 8 tiles its stencil overlaps (an
//                    atomic position per list); the same launch clears the
//                    field.
//   k_spread_tiles : blocks share the tiles, skip the empty ones, put a
//                    tile's list into marker order in shared memory and
//                    gather it.
// Work is proportional to the markers plus one write of the field.  Before, a
// block per tile scanned every marker (6252 markers on 96x80x72, 8640 tiles:
// 158 us of scans and 25 us of gathering by 512 threads per mostly empty
// tile; the whole call 227 us, now 61 us).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "../../include/turret.h"
#include "turret_internal.cuh"

using namespace turret;

namespace {

__device__ __forceinline__ float pk_in(float a) { return 0.125f * (3.0f - 2.0f * a + sqrtf(1.0f + 4.0f * a - 4.0f * a * a)); }
__device__ __forceinline__ float pk_out(float a) {
    return 0.125f * (5.0f - 2.0f * a - sqrtf(fmaxf(0.0f, -7.0f + 12.0f * a - 4.0f * a * a)));
}

// Stencil record of every marker from its position: base = floor(X) - 1 and
// the four 1-D Peskin weights per axis; h dS for the gather.  A stencil that
// leaves the grid (or a non-finite position) is parked at the origin with zero
// weights and flags *err.  tile_count (zero on entry) counts a tile's
// candidates, those beyond the list's capacity included.  Every thread also
// clears its share of the field (n4 float4 at an aligned address, then the
// last cells one by one).
__global__ void __launch_bounds__(128) k_records(int nm, const float *__restrict__ X, const float *__restrict__ h,
                                                 const float *__restrict__ dS, BoxGeom box, MRec *rec,
                                                 int *__restrict__ tile_list, int *__restrict__ tile_count, int cap,
                                                 int *err, float *__restrict__ field) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nm) {
        const int B[3] = {box.Bx, box.By, box.Bz};
        MRec r;
        int bv[3];
        bool bad = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float x = X[a * nm + k];
            const float fl = floorf(x);
            const float t = x - fl;
            int b = (int)fl - 1;
            float w4[4] = {pk_out(1.0f + t), pk_in(t), pk_in(1.0f - t), pk_out(2.0f - t)};
            if (!isfinite(x) || b < 0 || b > B[a] - 4) {
                b = 0;
                w4[0] = w4[1] = w4[2] = w4[3] = 0.0f;
                bad = true;
            }
            bv[a] = b;
            float *dst = (a == 0) ? r.wx : (a == 1) ? r.wy : r.wz;
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[q] = w4[q];
        }
        r.base = bv[0] | (bv[1] << 10) | (bv[2] << 20);
        const float d = bad ? 0.0f : dS[k];
        r.hdS[0] = h[k] * d;
        r.hdS[1] = h[nm + k] * d;
        r.hdS[2] = h[2 * nm + k] * d;
        rec[k] = r;
        if (bad) atomicMax(err, 1);
        // one or two tiles per axis; the positions of all are fetched together
        int tile[8], pos[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int x = bv[0] / TILE + (q & 1), y = bv[1] / TILE + (q >> 1 & 1), z = bv[2] / TILE + (q >> 2);
            const bool in = x <= (bv[0] + 3) / TILE && y <= (bv[1] + 3) / TILE && z <= (bv[2] + 3) / TILE;
            tile[q] = in ? x + box.tx * (y + box.ty * z) : -1;
            pos[q] = in ? atomicAdd(tile_count + tile[q], 1) : 0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (tile[q] >= 0) {
                if (pos[q] < cap) tile_list[(size_t)tile[q] * cap + pos[q]] = k;
                else atomicMax(err, 2);
            }
    }
    const long long total = 3 * box.nbox, step = (long long)gridDim.x * blockDim.x;
    if ((reinterpret_cast<uintptr_t>(field) & 15) == 0) {
        const long long n4 = total / 4;
        for (long long i = k; i < n4; i += step) reinterpret_cast<float4 *>(field)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (long long i = 4 * n4 + k; i < total; i += step) field[i] = 0.0f;
    } else {
        for (long long i = k; i < total; i += step) field[i] = 0.0f;
    }
}

// Gather of the non-empty tiles.  Block b looks at tiles b, b + gridDim.x, ...
// (the tiles of a surface are neighbours: the stride spreads them), ST_LOOK at
// a time, and gathers each that has candidates: its list is put into marker
// order (a thread per entry counts the smaller ones; a list holds some tens of
// markers, and beyond ST_THREADS, 2048 at most, it is sorted), then summed as in
// the time step's spreading: thread (cell c, slice q) sums slice q of each staged chunk, the
// slice sums are added in slice order.
constexpr int ST_SLICES = 8, ST_CELLS = TILE * TILE * TILE, ST_THREADS = ST_CELLS * ST_SLICES;
constexpr int ST_STAGE = 256, ST_LOOK = ST_THREADS;
constexpr int ST_BLOCKS = 152 * 4;  // four resident blocks per SM

// The cnt > ST_THREADS indices of a long list into ord in ascending order, by
// the whole block: bitonic sort, padded to a power of two; exchanges over less
// than a warp's width are shuffles.  (Ranked like a short list, 2000 markers in
// one cell of an 8^3 grid took 170 us a call, so 93; 1000 84 and 69.)
static_assert((MAX_CANDIDATES & (MAX_CANDIDATES - 1)) == 0, "the longest list fits its padding");
__device__ __forceinline__ void sort_list(const int *__restrict__ list, int cnt, int *ord) {
    const int tid = threadIdx.x;
    int n = 2 * ST_THREADS;
    while (n < cnt) n *= 2;
    // element i of a sequence sorted upwards where (i & run) is 0
    auto exchange = [](int i, int v, int run, int d) {
        const int o = __shfl_xor_sync(0xffffffffu, v, d);
        return ((i & run) == 0) == ((i & d) == 0) ? min(v, o) : max(v, o);
    };
    for (int i = tid; i < n; i += ST_THREADS) {
        int v = i < cnt ? __ldg(list + i) : 0x7fffffff;
        for (int run = 2; run <= 32; run *= 2)
            for (int d = run / 2; d > 0; d /= 2) v = exchange(i, v, run, d);
        ord[i] = v;
    }
    for (int run = 64; run <= n; run *= 2) {
        for (int d = run / 2; d >= 32; d /= 2) {
            __syncthreads();
            for (int i = tid; i < n / 2; i += ST_THREADS) {
                const int a = 2 * i - (i & (d - 1)), b = a + d;
                const int u = ord[a], v = ord[b];
                if ((u > v) == ((a & run) == 0)) {
                    ord[a] = v;
                    ord[b] = u;
                }
            }
        }
        __syncthreads();
        for (int i = tid; i < n; i += ST_THREADS) {
            int v = ord[i];
            for (int d = 16; d > 0; d /= 2) v = exchange(i, v, run, d);
            ord[i] = v;
        }
    }
}

__global__ void __launch_bounds__(ST_THREADS, 4) k_spread_tiles(BoxGeom box, const MRec *__restrict__ rec,
                                                             const int *__restrict__ tile_list,
                                                             const int *__restrict__ tile_count, int cap, int ntiles,
                                                             float *__restrict__ field) {
    __shared__ int s_tile[ST_LOOK], s_cnt[ST_LOOK], s_work;
    __shared__ __align__(16) int raw[MAX_CANDIDATES];
    __shared__ int ord[MAX_CANDIDATES];
    __shared__ int sbase[ST_STAGE];
    __shared__ float sw[12][ST_STAGE], sh[3][ST_STAGE];
    float *part = reinterpret_cast<float *>(raw);  // [ST_SLICES][3][ST_CELLS] once the list is ranked
    static_assert(ST_SLICES * 3 * ST_CELLS <= MAX_CANDIDATES, "partial sums reuse the unsorted list");
    const int tid = threadIdx.x, c = tid % ST_CELLS, q = tid / ST_CELLS;
    for (int first = blockIdx.x; first < ntiles; first += ST_LOOK * gridDim.x) {
        if (tid == 0) s_work = 0;
        __syncthreads();
        const long long mine = (long long)first + (long long)tid * gridDim.x;
        const int n_mine = mine < ntiles ? __ldg(tile_count + mine) : 0;
        if (n_mine > 0) {
            const int at = atomicAdd(&s_work, 1);  // the order of the tiles does not matter
            s_tile[at] = (int)mine;
            s_cnt[at] = min(n_mine, cap);
        }
        __syncthreads();
        const int work = s_work;
        for (int it = 0; it < work; ++it) {
            const int tile = s_tile[it], cnt = s_cnt[it];
            const int *list = tile_list + (size_t)tile * cap;
            if (cnt <= ST_THREADS) {
                const int k = tid < cnt ? __ldg(list + tid) : 0x7fffffff;
                raw[tid] = k;
                __syncthreads();
                if (tid < cnt) {
                    int r = 0;
                    for (int j = 0; j < cnt; j += 4) {
                        const int4 v = *reinterpret_cast<const int4 *>(raw + j);
                        r += (v.x < k) + (v.y < k) + (v.z < k) + (v.w < k);
                    }
                    ord[r] = k;
                }
            } else {
                sort_list(list, cnt, ord);
            }
            const int tx = tile % box.tx, ty = (tile / box.tx) % box.ty, tz = tile / (box.tx * box.ty);
            const int cx = TILE * tx + c % TILE, cy = TILE * ty + (c / TILE) % TILE, cz = TILE * tz + c / (TILE * TILE);
            float ax = 0.0f, ay = 0.0f, az = 0.0f;
            __syncthreads();
            for (int base = 0; base < cnt; base += ST_STAGE) {
                const int n = min(ST_STAGE, cnt - base);
                if (tid < n) {
                    const MRec r = rec[ord[base + tid]];
                    sbase[tid] = r.base;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        sw[e][tid] = r.wx[e];
                        sw[4 + e][tid] = r.wy[e];
                        sw[8 + e][tid] = r.wz[e];
                    }
                    sh[0][tid] = r.hdS[0];
                    sh[1][tid] = r.hdS[1];
                    sh[2][tid] = r.hdS[2];
                }
                __syncthreads();
                const int j0 = (n * q) / ST_SLICES, j1 = (n * (q + 1)) / ST_SLICES;
                for (int jj = j0; jj < j1; ++jj) {
                    const int pb = sbase[jj];
                    const int dx = cx - (pb & 1023), dy = cy - ((pb >> 10) & 1023), dz = cz - ((pb >> 20) & 1023);
                    if ((unsigned)dx < 4u && (unsigned)dy < 4u && (unsigned)dz < 4u) {
                        const float wv = sw[dx][jj] * sw[4 + dy][jj] * sw[8 + dz][jj];
                        ax = fmaf(wv, sh[0][jj], ax);
                        ay = fmaf(wv, sh[1][jj], ay);
                        az = fmaf(wv, sh[2][jj], az);
                    }
                }
                __syncthreads();
            }
            part[(q * 3 + 0) * ST_CELLS + c] = ax;
            part[(q * 3 + 1) * ST_CELLS + c] = ay;
            part[(q * 3 + 2) * ST_CELLS + c] = az;
            __syncthreads();
            if (tid < 3 * ST_CELLS) {
                const int a = tid / ST_CELLS;
                float v = 0.0f;
#pragma unroll
                for (int w = 0; w < ST_SLICES; ++w) v += part[(w * 3 + a) * ST_CELLS + c];
                if (cx < box.Bx && cy < box.By && cz < box.Bz)
                    field[a * box.nbox + ((size_t)cz * box.By + cy) * box.Bx + cx] = v;
            }
            __syncthreads();
        }
    }
}

struct SpreadLayout {
    BoxGeom box;
    int cap;
    size_t ntiles;
    size_t off_rec, off_list, off_count, off_err, bytes;
};

bool spread_layout(int32_t nx, int32_t ny, int32_t nz, int64_t nm, SpreadLayout &L) {
    if (nx < 4 || ny < 4 || nz < 4 || nx > 1023 || ny > 1023 || nz > 1023 || nm <= 0 || nm >= (1 << 24)) return false;
    L.box.Bx = nx;
    L.box.By = ny;
    L.box.Bz = nz;
    L.box.tx = (nx + TILE - 1) / TILE;
    L.box.ty = (ny + TILE - 1) / TILE;
    L.box.tz = (nz + TILE - 1) / TILE;
    L.box.nbox = (long long)nx * ny * nz;
    L.cap = (int)(nm < MAX_CANDIDATES ? nm : MAX_CANDIDATES);
    L.ntiles = (size_t)L.box.tx * L.box.ty * L.box.tz;
    size_t off = 0;
    auto take = [&](size_t b) {
        off = (off + 255) & ~(size_t)255;
        const size_t o = off;
        off += b;
        return o;
    };
    L.off_rec = take((size_t)nm * sizeof(MRec));
    take((size_t)nm * 4);  // unused; the fixed-scratch limit of ibm_spread_noalloc counts these bytes
    L.off_list = take(L.ntiles * (size_t)L.cap * 4);
    L.off_count = take(L.ntiles * 4);
    L.off_err = take(4);
    L.bytes = off;
    return true;
}

}  // namespace

// Enqueues the two kernels on the given scratch, waits for the stream and
// reads back the error word.
static turret_status run_spread(const float *X, const float *h, const float *dS, int64_t nm, int32_t nx, int32_t ny,
                                int32_t nz, float *field, char *scratch, const SpreadLayout &L, cudaStream_t s) {
    MRec *rec = (MRec *)(scratch + L.off_rec);
    int *list = (int *)(scratch + L.off_list);
    int *count = (int *)(scratch + L.off_count);
    int *err = (int *)(scratch + L.off_err);  // follows the counts
    if (cudaMemsetAsync(count, 0, L.off_err + 4 - L.off_count, s) != cudaSuccess) return TURRET_ECUDA;
    // a thread per marker, and enough threads to clear the field at the write bandwidth
    const long long clear = std::min<long long>((3 * L.box.nbox / 4 + 511) / 512, 152 * 16);
    const unsigned nb = (unsigned)std::max<long long>((nm + 127) / 128, clear);
    k_records<<<nb, 128, 0, s>>>((int)nm, X, h, dS, L.box, rec, list, count, L.cap, err, field);
    k_spread_tiles<<<(unsigned)std::min<size_t>(L.ntiles, ST_BLOCKS), ST_THREADS, 0, s>>>(L.box, rec, list, count, L.cap,
                                                                                      (int)L.ntiles, field);
    if (cudaGetLastError() != cudaSuccess) return TURRET_ECUDA;
    int herr = 0;
    if (cudaMemcpyAsync(&herr, err, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) return TURRET_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return TURRET_ECUDA;
    if (herr == 1) return TURRET_EDOMAIN;
    if (herr == 2) return TURRET_EOVERFLOW;
    return TURRET_OK;
}

extern "C" size_t ibm_spread_workspace_bytes(int32_t nx, int32_t ny, int32_t nz, int64_t n_markers) {
    SpreadLayout L;
    if (!spread_layout(nx, ny, nz, n_markers, L)) return 0;
    return L.bytes + 256;
}

extern "C" turret_status ibm_spread(const float *X, const float *h, const float *dS, int64_t n_markers, int32_t nx,
                                    int32_t ny, int32_t nz, float *field, void *workspace, size_t workspace_bytes,
                                    void *stream) {
    SpreadLayout L;
    if (!X || !h || !dS || !field || !spread_layout(nx, ny, nz, n_markers, L)) return TURRET_EINVAL;
    if (!workspace || workspace_bytes < L.bytes) return TURRET_ENOMEM;
    if (((uintptr_t)workspace & 255) != 0) return TURRET_EINVAL;
    return run_spread(X, h, dS, n_markers, nx, ny, nz, field, (char *)workspace, L, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// ibm_spread for callers that cannot allocate device memory.
//
// Some callers of this library may not call cudaMalloc at all: code that runs
// under a host framework whose memory pool owns the whole device, plugins that
// get no allocator from their host, and real-time loops that forbid
// allocation (and its implicit synchronisation) after start-up.  For them this
// entry point takes its scratch from a fixed array in the library's device
// image instead of a caller workspace.  The array is NOALLOC_SCRATCH_BYTES
// (8 MiB) and is held by every GPU that loads the library until the process
// exits.  The address of the array is a device address only on the device:
// host code obtains it once per device with cudaGetSymbolAddress (on the
// first call made with that device current) and passes it to the kernels.
// The cached address is valid for as long as the device's primary context
// lives: cudaDeviceReset unloads the image, and the entry point must not be
// called on that device afterwards.
constexpr size_t NOALLOC_SCRATCH_BYTES = (size_t)8 << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];
constexpr int NOALLOC_MAX_DEVICES = 64;
static std::mutex g_noalloc_mu;
static void *g_noalloc_ptr[NOALLOC_MAX_DEVICES];

extern "C" turret_status ibm_spread_noalloc(const float *X, const float *h, const float *dS, int64_t n_markers,
                                            int32_t nx, int32_t ny, int32_t nz, float *field, void *stream) {
    SpreadLayout L;
    if (!X || !h || !dS || !field || !spread_layout(nx, ny, nz, n_markers, L)) return TURRET_EINVAL;
    if (L.bytes > NOALLOC_SCRATCH_BYTES) return TURRET_ENOMEM;  // beyond the fixed scratch
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return TURRET_ECUDA;
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return TURRET_ECUDA;
            g_noalloc_ptr[dev] = p;
        }
        scratch = g_noalloc_ptr[dev];
    }
    // run_spread clears the counts and the error word first; records and listed
    // entries are rewritten by every call
    return run_spread(X, h, dS, n_markers, nx, ny, nz, field, (char *)scratch, L, (cudaStream_t)stream);
}
