// Cone-beam backprojection for FDK-OD (Sec. 2.2) and plain FDK (Sec. 2.1).
//
// For every square (a tile of 16 x 16 columns at a time), slab of slices and
// view, the detector window that the voxels touch is bounded by the tile's
// corners -- the column coordinate (Eq. 1 in square-local form) and the row
// coordinate z/U + (Nv-1)/2 are monotone in x, y and z -- and staged in shared
// memory, zero outside the detector; each thread adds U^-2 times the bilinear
// sample to the voxels of its column.  The gather is a sum over views of
// interpolated samples, not a dense contraction, so it runs on the FP32 pipes
// and the shared-memory path.  The kernels, in the order they are tried:
//   bp_pair_kernel (bp_pair.cuh): windows by TMA, two slabs per CTA; whole
//     volumes (a slab and its mirror image) and slabs of slices;
//   bp_generic_kernel: windows by plain loads, where TMA cannot describe the
//     source or a ring of the larger windows does not fit;
//   bp_global_kernel: no staging, where not even one window fits;
//   bp_persistent_kernel: a batch of plans in one launch.
//
// Two sources share each of them:
//   direct (D = 1 and the plain FDK baseline): Q_k itself, cropped per
//     (square, view) at crop = floor(phi + w0); column offset frac - w0;
//   decomposed (D > 1): the square's decimated data S'_q[j][v][t] at the
//     views beta_{jD}; column t = a - a_c - w0 (the second shift of
//     Sec. 2.1 folded into the addressing, as Sec. 2.2 says FDK-OD
//     interpolates once).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "bp_pair.cuh"
#include "fdkod_internal.cuh"
#include "tma.cuh"

namespace fdkod {
namespace {

constexpr int kWarps = kThreads / 32;

struct BpParams {
    const void *src;
    float *vol;
    const GeomEntry *geo;
    const int32_t *crop;
    const int32_t *w0;
    int *status;
    long long sq_stride, view_stride, row_stride;  // source layout (elements)
    int src_cols, src_rows;
    int row0;                // detector row held in the source's row 0
    int zoff, nz;            // slices zoff .. zoff + nz - 1, written to vol[z - zoff]
    int N, P, Nv, m, tps;    // tps: tiles per square side
    int nviews, vstep;       // views summed; table view index = j * vstep
    int Wd, Rw, J;           // staging window and views per chunk
    float scale;             // pi / nviews
};

__device__ __forceinline__ float ld_s(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ld_s(const __nv_bfloat16 *p) { return __bfloat162float(__ldg(p)); }
__device__ __forceinline__ float ld_s(const __half *p) { return __half2float(__ldg(p)); }

// One CTA of 16 x 16 threads owns a 16 x 16 column tile of one square and kZT
// consecutive slices, each thread one column's kZT voxels in registers; up to
// 8 views' windows are staged at a time.  WD: window columns at compile time
// (0: a.Wd), so that a sample's four loads take one address; a warp stages four
// rows of a window at a time, all their loads in flight together; the row
// coordinate's floor is one rounded-down addition.  253^3, 253 columns, 120 views,
// plain FDK: 3.63 ms before (row by row, every address and clamp per sample), 1.94.
template <typename TS, bool DIRECT, int WD>
__global__ void __launch_bounds__(kThreads, WD == 0 ? 1 : 3)
bp_generic_kernel(BpParams a) {
    extern __shared__ float win[];
    __shared__ float s_cb[kViewsPerChunk], s_sb[kViewsPerChunk], s_r[kViewsPerChunk], s_al[kViewsPerChunk],
        s_ga[kViewsPerChunk], s_g[kViewsPerChunk], s_toff[kViewsPerChunk], s_vrel[kViewsPerChunk];
    __shared__ int s_vlo[kViewsPerChunk], s_col0[kViewsPerChunk], s_skip[kViewsPerChunk];
    __shared__ long long s_off[kViewsPerChunk];

    const int tiles = a.tps * a.tps;
    const int q = blockIdx.x / tiles;
    const int tt = blockIdx.x - q * tiles;
    const int qy = q / a.m, qx = q - qy * a.m;
    int ix0, ix1, iy0, iy1;
    square_range(qx, a.m, a.N, ix0, ix1);
    square_range(qy, a.m, a.N, iy0, iy1);
    const int x0 = ix0 + (tt % a.tps) * kTile;
    const int y0 = iy0 + (tt / a.tps) * kTile;
    if (x0 > ix1 || y0 > iy1) return;  // ragged square: empty tile (uniform per CTA)
    const int xe = min(x0 + kTile - 1, ix1), ye = min(y0 + kTile - 1, iy1);
    const int z0 = a.zoff + blockIdx.y * kZT;
    const int z1 = min(z0 + kZT - 1, a.zoff + a.nz - 1);

    const float half_n = 0.5f * (float)(a.N - 1);
    const float xc = 0.5f * ((float)ix0 + (float)ix1) - half_n;  // square centre (exact half-integers)
    const float yc = 0.5f * ((float)iy0 + (float)iy1) - half_n;
    // centre of the full kZT-slice slab (also past the volume's end, so the
    // window always covers every slice the loop evaluates)
    const float zc = (float)z0 + 0.5f * (float)(kZT - 1) - half_n;
    const double vcd = 0.5 * (double)(a.Nv - 1);

    const int lx = threadIdx.x % kTile, ly = threadIdx.x / kTile;
    const int x = x0 + lx, y = y0 + ly;
    const bool active = x <= xe && y <= ye;
    const float dx = (float)x - half_n - xc, dy = (float)y - half_n - yc;
    constexpr float dz0 = -0.5f * (float)(kZT - 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wd = WD ? WD : a.Wd, WS = wd + 1;
    const int32_t w0q = a.w0[q];

    const uint32_t wbase = tma::smem_u32(win);
    float acc[kZT];
#pragma unroll
    for (int i = 0; i < kZT; ++i) acc[i] = 0.f;

    for (int jb = 0; jb < a.nviews; jb += a.J) {
        const int nj = min(a.J, a.nviews - jb);
        // 1. per-view window, one warp per view, lanes 0..7 take the corners
        if (warp < nj) {
            const int j = jb + warp;
            const int k = j * a.vstep;
            const size_t o = (size_t)q * a.P + k;
            const GeomEntry ge = a.geo[o];
            const float gf = ge.g_hi;
            const float toff = DIRECT ? ge.frac - (float)w0q : -(float)w0q;
            const int c = lane & 7;
            const float cx = (float)((c & 1) ? xe : x0) - half_n - xc;
            const float cy = (float)((c & 2) ? ye : y0) - half_n - yc;
            const float cz = (c & 4) ? -dz0 : dz0;
            const float dd = fmaf(ge.cb, cx, ge.sb * cy);
            const float invU = gf / fmaf(ge.r, dd, 1.0f);
            const float t = fmaf(invU, fmaf(ge.alpha, cx, ge.gamma * cy), toff);
            const float zq = zc * ge.r * dd;
            const double vcen = fma((double)zc, (double)ge.g_hi + (double)ge.g_lo, vcd);
            const double v = vcen + (double)(invU * (cz - zq));
            float tmin = t, tmax = t;
            double vmin = v, vmax = v;
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) {
                tmin = fminf(tmin, __shfl_xor_sync(0xffffffffu, tmin, off));
                tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, off));
                vmin = fmin(vmin, __shfl_xor_sync(0xffffffffu, vmin, off));
                vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, off));
            }
            if (lane == 0) {
                const int tlo = (int)floorf(tmin) - 1;
                const int vlo = (int)floor(vmin) - 1;
                // a window too small is reported and its view left out
                const int skip = (int)floorf(tmax) + 2 - tlo > wd - 1 || (int)floor(vmax) + 2 - vlo > a.Rw - 1;
                if (skip) atomicOr(a.status, 1);
                s_skip[warp] = skip;
                s_cb[warp] = ge.cb;
                s_sb[warp] = ge.sb;
                s_r[warp] = ge.r;
                s_al[warp] = ge.alpha;
                s_ga[warp] = ge.gamma;
                s_g[warp] = gf;
                s_toff[warp] = toff - (float)tlo;
                s_vrel[warp] = (float)(vcen - (double)vlo);
                s_vlo[warp] = vlo;
                if (DIRECT) {
                    const int col0 = a.crop[o] + tlo;
                    s_col0[warp] = col0;
                    s_off[warp] = (long long)k * a.view_stride + col0;
                } else {
                    s_col0[warp] = tlo;
                    s_off[warp] = (long long)q * a.sq_stride + (long long)j * a.view_stride + tlo;
                }
            }
        }
        __syncthreads();
        // 2. stage the windows: a warp takes rows warp, warp + kWarps, ... of
        // each, kRows at a time, lanes along columns
        const TS *src = (const TS *)a.src;
        constexpr int kRows = 4, kCols = WD ? (WD + 31) / 32 : 1;
        for (int w = 0; w < nj; ++w) {
            const TS *vw = src + s_off[w];
            const int col0 = s_col0[w], r0 = s_vlo[w] - a.row0;  // row of the source in window row 0
            float *dst = win + (size_t)w * a.Rw * WS;
            for (int cb = 0; cb < wd; cb += 32 * kCols)
                for (int rb = warp; rb < a.Rw; rb += kRows * kWarps) {
                    float val[kRows][kCols];
#pragma unroll
                    for (int u = 0; u < kRows; ++u) {
                        const int r = rb + u * kWarps, v = r0 + r;
                        const bool rok = r < a.Rw && v >= 0 && v < a.src_rows;
#pragma unroll
                        for (int i = 0; i < kCols; ++i) {
                            const int c = cb + 32 * i + lane, col = col0 + c;
                            val[u][i] = rok && c < wd && col >= 0 && col < a.src_cols
                                            ? ld_s(vw + (long long)v * a.row_stride + c) : 0.f;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kRows; ++u)
#pragma unroll
                        for (int i = 0; i < kCols; ++i) {
                            const int r = rb + u * kWarps, c = cb + 32 * i + lane;
                            if (r < a.Rw && c < wd) dst[r * WS + c] = val[u][i];
                        }
                }
        }
        __syncthreads();
        // 3. accumulate
        if (active) {
            for (int w = 0; w < nj; ++w) {
                if (s_skip[w]) continue;
                const float dd = fmaf(s_cb[w], dx, s_sb[w] * dy);
                const float invU = s_g[w] / fmaf(s_r[w], dd, 1.0f);
                const float t = fmaf(invU, fmaf(s_al[w], dx, s_ga[w] * dy), s_toff[w]);
                const float tf = floorf(t);
                const float wgt = invU * invU;
                const float a1 = wgt * (t - tf), a0 = wgt - a1;
                const float zq = zc * s_r[w] * dd;
                const float vb = fmaf(-invU, zq, s_vrel[w]);
                // byte address of window row r, this column: r 4 WS + base (the
                // floor's bits carry kFloorBits)
                const uint32_t base = wbase + 4u * ((uint32_t)(w * a.Rw) * (uint32_t)WS + (uint32_t)(int)tf) -
                                      kFloorBits * (4u * (uint32_t)WS);
#pragma unroll
                for (int i = 0; i < kZT; ++i) {
                    const float v = fmaf(invU, dz0 + (float)i, vb);
                    const float vm = floor_biased(v);
                    const float fv = v - (vm - kFloorBias);
                    const uint32_t ad = __float_as_uint(vm) * (4u * (uint32_t)WS) + base;
                    const uint32_t ad2 = WD ? ad : ad + 4u * (uint32_t)WS;
                    constexpr int kNext = WD ? 4 * (WD + 1) : 0;
                    const float c0 = fmaf(a1, Lds<float, 4>::f(ad), a0 * Lds<float, 0>::f(ad));
                    const float c1 = fmaf(a1, Lds<float, kNext + 4>::f(ad2), a0 * Lds<float, kNext>::f(ad2));
                    acc[i] = fmaf(fv, c1 - c0, acc[i] + c0);
                }
            }
        }
        __syncthreads();
    }
    if (active) {
#pragma unroll
        for (int i = 0; i < kZT; ++i)
            if (z0 + i <= z1) a.vol[((size_t)(z0 + i - a.zoff) * a.N + y) * a.N + x] = acc[i] * a.scale;
    }
}

// Unstaged form for windows too large to stage in shared memory (a source
// close to the volume magnifies a tile's footprint on the detector): the
// same tiling and arithmetic as bp_generic_kernel, every sample read from the
// source in global memory (zero outside it).  Row coordinates stay relative
// to an integer base row per view, as in the staged kernels.
template <typename TS, bool DIRECT>
__global__ void __launch_bounds__(kThreads)
bp_global_kernel(BpParams a) {
    const int tiles = a.tps * a.tps;
    const int q = blockIdx.x / tiles;
    const int tt = blockIdx.x - q * tiles;
    const int qy = q / a.m, qx = q - qy * a.m;
    int ix0, ix1, iy0, iy1;
    square_range(qx, a.m, a.N, ix0, ix1);
    square_range(qy, a.m, a.N, iy0, iy1);
    const int x0 = ix0 + (tt % a.tps) * kTile;
    const int y0 = iy0 + (tt / a.tps) * kTile;
    if (x0 > ix1 || y0 > iy1) return;
    const int xe = min(x0 + kTile - 1, ix1), ye = min(y0 + kTile - 1, iy1);
    const int z0 = a.zoff + blockIdx.y * kZT;
    const int z1 = min(z0 + kZT - 1, a.zoff + a.nz - 1);
    const float half_n = 0.5f * (float)(a.N - 1);
    const float xc = 0.5f * ((float)ix0 + (float)ix1) - half_n;
    const float yc = 0.5f * ((float)iy0 + (float)iy1) - half_n;
    const float zc = 0.5f * ((float)z0 + (float)z1) - half_n;
    const double vcd = 0.5 * (double)(a.Nv - 1);
    const int lx = threadIdx.x % kTile, ly = threadIdx.x / kTile;
    const int x = x0 + lx, y = y0 + ly;
    if (x > xe || y > ye) return;  // no block barrier below
    const float dx = (float)x - half_n - xc, dy = (float)y - half_n - yc;
    const float dz0 = (float)z0 - half_n - zc;
    const int32_t w0q = a.w0[q];
    const TS *src = (const TS *)a.src;
    auto at = [&](long long off, int r, int c) -> float {  // sample (row r of the detector, column c of the source)
        const int rr = r - a.row0;
        return (rr >= 0 && rr < a.src_rows && c >= 0 && c < a.src_cols) ? ld_s(src + off + (long long)rr * a.row_stride + c)
                                                                         : 0.f;
    };
    float acc[kZT];
#pragma unroll
    for (int i = 0; i < kZT; ++i) acc[i] = 0.f;
    for (int j = 0; j < a.nviews; ++j) {
        const int k = j * a.vstep;
        const size_t o = (size_t)q * a.P + k;
        const GeomEntry ge = a.geo[o];
        const float toff = DIRECT ? ge.frac - (float)w0q : -(float)w0q;
        const float dd = fmaf(ge.cb, dx, ge.sb * dy);
        const float invU = ge.g_hi / fmaf(ge.r, dd, 1.0f);
        const float t = fmaf(invU, fmaf(ge.alpha, dx, ge.gamma * dy), toff);
        const float tf = floorf(t);
        const float ft = t - tf;
        const int col = (DIRECT ? a.crop[o] : 0) + (int)tf;
        const long long off = DIRECT ? (long long)k * a.view_stride : (long long)q * a.sq_stride + (long long)j * a.view_stride;
        const float wgt = invU * invU;
        const double vcen = fma((double)zc, (double)ge.g_hi + (double)ge.g_lo, vcd);
        const int vbase = (int)floor(vcen);
        const float zq = zc * ge.r * dd;
        const float vb = fmaf(-invU, zq, (float)(vcen - (double)vbase));
#pragma unroll
        for (int i = 0; i < kZT; ++i) {
            const float v = fmaf(invU, dz0 + (float)i, vb);
            const float vf = floorf(v);
            const float fv = v - vf;
            const int r = vbase + (int)vf;
            const float s00 = at(off, r, col), s01 = at(off, r, col + 1);
            const float s10 = at(off, r + 1, col), s11 = at(off, r + 1, col + 1);
            const float c0 = fmaf(ft, s01 - s00, s00);
            const float c1 = fmaf(ft, s11 - s10, s10);
            acc[i] = fmaf(wgt, fmaf(fv, c1 - c0, c0), acc[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < kZT; ++i)
        if (z0 + i <= z1) a.vol[((size_t)(z0 + i - a.zoff) * a.N + y) * a.N + x] = acc[i] * a.scale;
}

template <typename TS, bool DIRECT, int WD>
cudaError_t launch_generic(BpParams prm, int nsq, cudaStream_t st) {
    const size_t smem = sizeof(float) * (size_t)prm.J * prm.Rw * ((WD ? WD : prm.Wd) + 1);
    cudaError_t e = ensure_smem<bp_generic_kernel<TS, DIRECT, WD>>(smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(nsq * prm.tps * prm.tps), (unsigned)((prm.nz + kZT - 1) / kZT));
    bp_generic_kernel<TS, DIRECT, WD><<<grid, kThreads, smem, st>>>(prm);
    return cudaGetLastError();
}

// Views per chunk for windows of `cols` columns: as many as three CTAs per SM
// leave room for, at least two; 0 where they do not fit.
int generic_views(const BpParams &prm, int cols) {
    const size_t per_view = sizeof(float) * (size_t)prm.Rw * (cols + 1);
    const int j = (int)std::min<size_t>(kViewsPerChunk, (72u * 1024u) / per_view);
    return j >= 2 ? j : 0;
}

template <typename TS, bool DIRECT>
cudaError_t launch_t(BpParams prm, int nsq, cudaStream_t st) {
    if (prm.J < 1) {  // one view's window does not fit shared memory: sample from global memory
        dim3 grid((unsigned)(nsq * prm.tps * prm.tps), (unsigned)((prm.nz + kZT - 1) / kZT));
        bp_global_kernel<TS, DIRECT><<<grid, kThreads, 0, st>>>(prm);
        return cudaGetLastError();
    }
    const int cols = prm.Wd <= 32 ? 32 : prm.Wd <= 48 ? 48 : prm.Wd <= 64 ? 64 : 0;
    const int j = cols ? generic_views(prm, cols) : 0;
    if (j > 0) {
        prm.J = j;
        switch (cols) {
            case 32: return launch_generic<TS, DIRECT, 32>(prm, nsq, st);
            case 48: return launch_generic<TS, DIRECT, 48>(prm, nsq, st);
            default: return launch_generic<TS, DIRECT, 64>(prm, nsq, st);
        }
    }
    return launch_generic<TS, DIRECT, 0>(prm, nsq, st);
}

// Parameters of one plan in the batch's persistent launch.
struct BpTmaParams {
    float *vol;
    const GeomEntry *geo;
    const int32_t *crop;
    const int32_t *w0;
    int *status;
    int N, P, Nv, m, tps;
    int nviews, vstep, Pd;
    int RW, tile_stride;  // window rows; elements per staged window (128-byte multiple)
    int row0;             // detector row held in the source's row 0
    int zoff, nz;         // slices zoff .. zoff + nz - 1, written to vol[z - zoff]
    float scale;
};

// address bias: (row + kMagicBits) * 4 WD wraps to row * 4 WD in 32 bits once
// tbase absorbs -kMagicBits * 4 WD (keeps the unsigned arithmetic explicit)
constexpr int kMagicBits = 0x4B400000;
// ---------------------------------------------------------------------------
// Persistent form for a batch of plans (float32 windows): one launch, as
// many CTAs as fit the GPU, each taking work items (plan, tile, z-slab) from
// an atomic counter until the list is exhausted.  Same tiling as the generic
// kernel; each view's window is one 3D bulk-tensor copy (zero fill outside
// the source), two stages of kViewsPerStage views are in flight (the copy of
// stage c + 1 overlaps the gather of stage c), the per-view set-up is FP32
// only, and per slice: v = fma(1/U, i, v0), floor, fraction, one multiply-add
// for the row address, four shared loads, two column lerps pre-weighted by
// U^-2, row lerp.  The plan's tensor map and parameters are read from global
// memory and the window width is a run-time value (the second window row is
// one add away).  The mbarrier stages continue from item to item; waits on
// the copies are bounded (FDKOD_ERR_TIMEOUT, then drain and exit).
struct BatchInst {
    BpTmaParams a;
    int direct, WD;
};

__global__ void __launch_bounds__(kThreads, 3)
bp_persistent_kernel(const CUtensorMap *__restrict__ maps, const BatchInst *__restrict__ insts,
                     const int4 *__restrict__ items, int nitems, int *counter) {
    constexpr int kAl = 4;  // float windows: 16-byte copy alignment in elements
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *sm = (float *)(smem_raw + ((128u - (tma::smem_u32(smem_raw) & 127u)) & 127u));
    const uint32_t sbase = tma::smem_u32(sm);
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ float4 s_pa[2][kViewsPerStage];
    __shared__ float4 s_pb[2][kViewsPerStage];
    __shared__ float s_zcr[2][kViewsPerStage];
    __shared__ int s_tx[2][kViewsPerStage], s_ty[2][kViewsPerStage], s_tz[2][kViewsPerStage];
    __shared__ int s_skip[2][kViewsPerStage];
    __shared__ int s_item;
    if (threadIdx.x == 0) {
        tma::mbar_init(&bars[0], 1);
        tma::mbar_init(&bars[1], 1);
        tma::fence_mbar_init();
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t gc = 0;  // chunks this CTA has run: stage gc % 2, parity (gc / 2) % 2

    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= nitems) break;
        const int4 it = items[item];  // plan, tile, z-slab
        const BpTmaParams a = insts[it.x].a;
        const bool direct = insts[it.x].direct != 0;
        const int WD = insts[it.x].WD;
        const CUtensorMap *map = maps + it.x;

        const int tiles = a.tps * a.tps;
        const int q = it.y / tiles;
        const int tt = it.y - q * tiles;
        const int qy = q / a.m, qx = q - qy * a.m;
        int ix0, ix1, iy0, iy1;
        square_range(qx, a.m, a.N, ix0, ix1);
        square_range(qy, a.m, a.N, iy0, iy1);
        const int x0 = ix0 + (tt % a.tps) * kTile;
        const int y0 = iy0 + (tt / a.tps) * kTile;
        if (x0 > ix1 || y0 > iy1) continue;  // ragged square: empty tile (uniform)
        const int xe = min(x0 + kTile - 1, ix1), ye = min(y0 + kTile - 1, iy1);
        const int z0 = a.zoff + it.z * kZT;
        const int z1 = min(z0 + kZT - 1, a.zoff + a.nz - 1);
        const float half_n = 0.5f * (float)(a.N - 1);
        const float xc = 0.5f * ((float)ix0 + (float)ix1) - half_n;
        const float yc = 0.5f * ((float)iy0 + (float)iy1) - half_n;
        const float zc = (float)z0 + 0.5f * (float)(kZT - 1) - half_n;
        const float vcd = 0.5f * (float)(a.Nv - 1);
        const int lx = threadIdx.x % kTile, ly = threadIdx.x / kTile;
        const int x = x0 + lx, y = y0 + ly;
        const bool active = x <= xe && y <= ye;
        const float dx = (float)x - half_n - xc, dy = (float)y - half_n - yc;
        const int32_t w0q = a.w0[q];
        const int nch = (a.nviews + kViewsPerStage - 1) / kViewsPerStage;

        auto setup = [&](int c, int st) {
            const int nj = min(kViewsPerStage, a.nviews - c * kViewsPerStage);
            if (warp < nj) {
                const int j = c * kViewsPerStage + warp;
                const int k = j * a.vstep;
                const size_t o = (size_t)q * a.P + k;
                const GeomEntry ge = a.geo[o];
                const int cbase = direct ? a.crop[o] : 0;
                const float toff = direct ? ge.frac - (float)w0q : -(float)w0q;
                const int cc = lane & 7;
                const float cx = (float)((cc & 1) ? xe : x0) - half_n - xc;
                const float cy = (float)((cc & 2) ? ye : y0) - half_n - yc;
                const float cz = (cc & 4) ? 0.5f * (float)(kZT - 1) : -0.5f * (float)(kZT - 1);
                const float dd = fmaf(ge.cb, cx, ge.sb * cy);
                const float invU = __fdividef(ge.g_hi, fmaf(ge.r, dd, 1.0f));
                const float t = fmaf(invU, fmaf(ge.alpha, cx, ge.gamma * cy), toff);
                const float zcr = zc * ge.r;
                const float ph = zc * ge.g_hi;
                const float pl = fmaf(zc, ge.g_lo, fmaf(zc, ge.g_hi, -ph));
                const float v = (ph + vcd) + (pl + invU * (cz - zcr * dd));
                float tmin = t, tmax = t, vmin = v, vmax = v;
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) {
                    tmin = fminf(tmin, __shfl_xor_sync(0xffffffffu, tmin, off));
                    tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, off));
                    vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, off));
                    vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, off));
                }
                if (lane == 0) {
                    const int clo = cbase + (int)floorf(tmin) - 1;
                    const int chi = cbase + (int)floorf(tmax) + 2;
                    const int xs = clo & ~(kAl - 1);
                    const int vlo = (int)floorf(vmin) - 1;
                    const int vhi = (int)floorf(vmax) + 2;
                    const int skip = (chi - xs > WD - 1) || (vhi - vlo > a.RW - 1);
                    if (skip) atomicOr(a.status, 1);
                    s_pa[st][warp] = make_float4(ge.cb, ge.sb, ge.r, ge.alpha);
                    s_pb[st][warp] = make_float4(ge.gamma, ge.g_hi, toff - (float)(xs - cbase),
                                                 (ph - ((float)vlo - vcd)) + pl);
                    s_zcr[st][warp] = zcr;
                    s_tx[st][warp] = xs;
                    s_ty[st][warp] = vlo - a.row0;
                    s_tz[st][warp] = direct ? k : q * a.Pd + j;
                    s_skip[st][warp] = skip;
                }
            }
        };
        auto issue = [&](int c, int st) {
            const int nj = min(kViewsPerStage, a.nviews - c * kViewsPerStage);
            tma::fence_proxy_async();
            tma::mbar_arrive_expect_tx(&bars[st], (uint32_t)(nj * a.RW * WD * 4));
            for (int w = 0; w < nj; ++w)
                tma::load_3d(sm + (size_t)(st * kViewsPerStage + w) * a.tile_stride, map, &bars[st], s_tx[st][w],
                             s_ty[st][w], s_tz[st][w]);
        };

        setup(0, (int)(gc & 1u));
        __syncthreads();
        if (threadIdx.x == 0) issue(0, (int)(gc & 1u));
        float acc[kZT];
#pragma unroll
        for (int i = 0; i < kZT; ++i) acc[i] = 0.f;
        const uint32_t rowb = 4u * (uint32_t)WD;
        for (int c = 0; c < nch; ++c) {
            const uint32_t g = gc + (uint32_t)c;
            const int st = (int)(g & 1u);
            if (c + 1 < nch) setup(c + 1, st ^ 1);
            __syncthreads();
            if (c + 1 < nch && threadIdx.x == 0) issue(c + 1, st ^ 1);
            const bool ok = tma::mbar_wait_bounded(&bars[st], (g >> 1) & 1u, kWaitLimitNs);
            if (!__syncthreads_and(ok)) {
                if (threadIdx.x == 0) atomicOr(a.status, 2);
                tma::mbar_wait_bounded(&bars[st], (g >> 1) & 1u, kWaitLimitNs);
                if (c + 1 < nch) tma::mbar_wait_bounded(&bars[st ^ 1], ((g + 1) >> 1) & 1u, kWaitLimitNs);
                return;
            }
            if (active) {
                const int nj = min(kViewsPerStage, a.nviews - c * kViewsPerStage);
                for (int w = 0; w < nj; ++w) {
                    if (s_skip[st][w]) continue;
                    const float4 pa = s_pa[st][w];
                    const float4 pb = s_pb[st][w];
                    const float dd = fmaf(pa.x, dx, pa.y * dy);
                    const float invU = __fdividef(pb.y, fmaf(pa.z, dd, 1.0f));
                    const float t = fmaf(invU, fmaf(pa.w, dx, pb.x * dy), pb.z);
                    const float tf = floorf(t);
                    const float wgt = invU * invU;
                    const float a1 = wgt * (t - tf);
                    const float a0 = wgt - a1;
                    const float vb0 = fmaf(invU, -0.5f * (float)(kZT - 1) - s_zcr[st][w] * dd, pb.w);
                    const uint32_t tbase = sbase + 4u * ((uint32_t)(st * kViewsPerStage + w) *
                                                             (uint32_t)a.tile_stride + (uint32_t)(int)tf) -
                                           (uint32_t)kMagicBits * rowb;
#pragma unroll
                    for (int i = 0; i < kZT; ++i) {
                        const float v = fmaf(invU, (float)i, vb0);
                        const float fl = floorf(v);
                        const float fv = v - fl;
                        const uint32_t ad = (uint32_t)((int)fl + kMagicBits) * rowb + tbase;
                        const uint32_t ad2 = ad + rowb;
                        const float c0 = fmaf(a1, Lds<float, 4>::f(ad), a0 * Lds<float, 0>::f(ad));
                        const float c1 = fmaf(a1, Lds<float, 4>::f(ad2), a0 * Lds<float, 0>::f(ad2));
                        acc[i] = fmaf(fv, c1 - c0, acc[i] + c0);
                    }
                }
            }
            __syncthreads();
        }
        gc += (uint32_t)nch;
        if (active) {
#pragma unroll
            for (int i = 0; i < kZT; ++i)
                if (z0 + i <= z1) a.vol[((size_t)(z0 + i - a.zoff) * a.N + y) * a.N + x] = acc[i] * a.scale;
        }
    }
}

// Tensor map of a source (Q itself, or the decomposed data, float32) that
// holds `rows` detector rows, with boxes of WD columns x `box_rows` rows.
// False where TMA cannot describe it: the source must be 16-byte aligned, its
// rows whole 16-byte units, and the window must fit a box (WD != 0, <= 256
// rows).
bool source_map(const PlanImpl &p, const SquareSet &ss, bool direct, const void *src, int rows, int WD, int box_rows,
                CUtensorMap &map) {
    const int es = (direct && p.qtype != FDKOD_F32) ? 2 : 4;
    if (WD == 0 || box_rows > 256 || ((uintptr_t)src & 15) != 0) return false;
    if (direct && ((size_t)p.g.Nu * es) % 16 != 0) return false;
    const uint64_t cols = direct ? (uint64_t)p.g.Nu : (uint64_t)p.Tstride;
    const uint64_t dims[3] = {cols, (uint64_t)rows, direct ? (uint64_t)p.g.P : (uint64_t)ss.nsq * p.Pd};
    const uint64_t strides[2] = {cols * es, cols * es * (uint64_t)rows};
    const uint32_t box[3] = {(uint32_t)WD, (uint32_t)box_rows, 1u};
    const CUtensorMapDataType dt = es == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : (p.qtype == FDKOD_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                           : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
    return encode_map_3d(&map, dt, src, dims, strides, box) == cudaSuccess;
}

// Tensor map, parameters and window width of a plan in the batch's persistent
// launch (float32 windows; it has no test hooks); false when it cannot take it.
bool make_tma_launch(const PlanImpl &p, const SquareSet &ss, bool direct, const void *src, float *vol,
                     const Band &b, CUtensorMap &map, BpTmaParams &a, int &WD) {
    WD = ss.WdT;
    if (!source_map(p, ss, direct, src, b.nrows, WD, ss.Rw, map)) return false;
    a = BpTmaParams{};
    a.vol = vol;
    a.geo = ss.geo;
    a.crop = ss.crop;
    a.w0 = ss.w0;
    a.status = p.status;
    a.N = p.g.N;
    a.P = p.g.P;
    a.Nv = p.g.Nv;
    a.m = ss.m;
    a.tps = ss.tiles_per_side;
    a.Pd = p.Pd;
    a.RW = ss.Rw;
    a.row0 = b.row0;
    a.zoff = b.zoff;
    a.nz = b.nz;
    a.tile_stride = pair_tile_stride(4, ss.Rw, WD);  // elements per staged window, a 128-byte multiple
    if (direct) {
        a.nviews = p.g.P;
        a.vstep = 1;
        a.scale = (float)(M_PI / (double)p.g.P);
    } else {
        a.nviews = p.Pd;
        a.vstep = p.D;
        a.scale = (float)(M_PI / (double)p.Pd);
    }
    return true;
}

// opt-in shared memory per block of the current device, less room for the
// kernels' static shared memory; *per_sm: the SM's shared memory less what
// the runtime reserves per block, shared by the CTAs of an SM
size_t smem_budget(size_t *per_sm = nullptr) {
    int dev = 0, optin = 0, sm = 0, reserved = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess)
        return 0;
    if (per_sm) *per_sm = (size_t)sm;
    return optin > 2048 ? (size_t)optin - 2048 : 0;
}

// Ring of the pair kernel for windows of `rows` x WD elements of es bytes: 3
// slots of 2 views, or 2 of 2, where the SM then holds the CTAs that the
// registers allow (each with its static shared memory and the runtime's
// reserve, 2 KiB together at most), else 3 of 1 if one CTA fits; false if not.
// (250^3, R = 2.5 N: 3 x 1 views 917 us, 2 x 2 846; 512^3: 3 x 2 8.35 ms, 2 x 2
// 8.38; all four 1-2 % less since warps outside a tile take no part.)
bool pair_ring(int es, int zp, int rows, PairShape &s) {
    size_t per_sm = 0;
    const size_t budget = smem_budget(&per_sm);
    const int ts = pair_tile_stride(es, rows, s.WD);
    s.vps = 2;
    for (s.slots = 3; s.slots >= 2; --s.slots)
        if ((size_t)pair_ctas(zp) * (pair_smem(es, 2, s.slots, ts) + 2048) <= per_sm) return true;
    s.vps = 1;
    s.slots = 3;
    return pair_smem(es, 1, 3, ts) <= budget;
}

// CTAs of the pair kernel that an SM holds at once: the registers' count, or
// what the ring leaves room for
int pair_resident(int es, int zp, int rows, const PairShape &s) {
    size_t per_sm = 0;
    smem_budget(&per_sm);
    const size_t smem = pair_smem(es, s.vps, s.slots, pair_tile_stride(es, rows, s.WD)) + 2048;
    return std::max(1, (int)std::min<size_t>((size_t)pair_ctas(zp), per_sm / smem));
}

// What rounds in the pair kernel's shape for `pairs` pairs of slices per column
// (slices per slab, CTAs that share the views), with the ring of s.WD columns;
// false where the windows are too large to stage.  32
// pairs per thread halve the per-view set-up and stage fewer margin rows
// (512^3: 8.25 ms against 8.61 at 16), but need enough CTAs: 2 per SM, half as
// many of them (from 160^3 to 256^3 both take the same time within 4 %), and
// they must not compute much more than they keep (the last slab's excess).
bool pair_slabs(const PlanImpl &p, const SquareSet &ss, bool direct, bool mirror, int pairs, PairShape &s) {
    const int es = (direct && p.qtype != FDKOD_F32) ? 2 : 4;
    s.nsplit = 1;
    const long long tiles = (long long)ss.nsq * ss.tiles_per_side * ss.tiles_per_side;
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int n32 = (pairs + 31) / 32, n16 = (pairs + 15) / 16;
    // 16-bit windows: only far sources and 16 waves of CTAs (512^3 x 180 bf16, R = 6 N:
    // 9.61 ms, 9.78 with 16 slices; R = 3 N 10.56, 10.40; R = 2 N 11.9, 11.0; 256^3 x
    // 90 f16, R = 4 N 722 us, 692).
    const bool far = es == 4 || ss.drift < 0.25;
    s.zp = 32;
    if (far && ss.Rw <= 256 && tiles * n32 >= (es == 4 ? 2LL : 16LL) * pair_ctas(32) * sms && 64 * n32 <= 34 * n16 &&
        pair_ring(es, 32, ss.Rw, s) && s.vps == 2)
        return true;
    s.zp = 16;
    if (ss.Rw2 > 256 || !pair_ring(es, 16, ss.Rw2, s)) return false;
    // Clusters share the views where the tiles leave SMs idle: as many CTAs as
    // fit the GPU at once, at least 5 views each (64^3 x 45 views, 32 CTAs: 36.4
    // us alone, 16.8 in clusters of 8; 96^3 x 67, 108 CTAs: 51.7, 37.3 in 4,
    // 44.9 in 8).  Up to two waves, smaller pieces still fill the last wave
    // better where they are long enough (128^3 x 64, 256 CTAs: 74.3, 69.4 in 4;
    // x 179: 196, 167; 160^3 x 55, 500 CTAs: 115, 109 in 2), but not beyond
    // (192^3 x 67, 864 CTAs: 203, 211 in 2).  What fits at once is what the ring
    // leaves room for: with R = 1.2 N one CTA per SM, where 128^3 x 64 takes 162 us
    // alone, 227 in 4, and a second wave does not pay (96^3 x 67, 108 CTAs: 107, 113
    // in 4).
    if (mirror) {
        const int views = direct ? p.g.P : p.Pd;
        const int resident = pair_resident(es, 16, ss.Rw2, s);
        const long long ctas = tiles * n16, slots = (long long)resident * sms;
        for (int n = 8; n >= 2 && s.nsplit == 1; n /= 2)
            if (ctas * n <= slots && views >= 5 * n) s.nsplit = n;
        if (s.nsplit < 4 && resident > 1 && ctas * 4 <= 3 * slots && views >= 64) s.nsplit = 4;
        if (s.nsplit == 1 && resident > 1 && ctas * 4 <= 5 * slots && views >= 32) s.nsplit = 2;
    }
    return true;
}

// The pair kernel's shape; false where it does not apply (no window width, or
// windows too large to stage).  The narrowest window decides what rounds, so
// that a wider one chosen by fdkod_set_tile gives the same result; it is
// taken where the shape has a ring of its width (512^3: up to 64 columns with
// 32 slices per slab; 16 slices would fit 96, and round otherwise).
bool pair_shape(const PlanImpl &p, const SquareSet &ss, bool direct, bool mirror, int pairs, PairShape &s) {
    const int es = (direct && p.qtype != FDKOD_F32) ? 2 : 4;
    s.mirror = mirror;
    s.WD = window_width(es == 4 ? ss.need : ss.need16);
    if (s.WD == 0 || !pair_slabs(p, ss, direct, mirror, pairs, s)) return false;
    PairShape wide = s;
    wide.WD = es == 4 ? ss.WdT : ss.WdT16;
    if (wide.WD != s.WD && pair_ring(es, s.zp, s.zp == 32 ? ss.Rw : ss.Rw2, wide) && (s.zp == 16 || wide.vps == 2))
        s = wide;
    return true;
}

// The staged kernel over the slices of b (mirror: over the whole detector and
// the slice pairs p0 .. p1 - 1, i.e. slices p and N - 1 - p, of the whole
// volume, with the shape s of the whole launch).
cudaError_t try_launch_pair(const PlanImpl &p, const SquareSet &ss, bool direct, const void *src, float *vol,
                            cudaStream_t st, const PairShape &s, const Band &b, int p0, int p1, bool &launched) {
    launched = false;
    const int es = (direct && p.qtype != FDKOD_F32) ? 2 : 4;
    const int rows = s.zp == 32 ? ss.Rw : ss.Rw2;
    CUtensorMap map;
    if (!source_map(p, ss, direct, src, b.nrows, s.WD, rows, map)) return cudaSuccess;
    BpPairParams a{};
    a.vol = vol;
    a.geo = ss.geo;
    a.crop = ss.crop;
    a.w0 = ss.w0;
    a.status = p.status;
    a.N = p.g.N;
    a.P = p.g.P;
    a.Nv = p.g.Nv;
    a.m = ss.m;
    a.tps = ss.tiles_per_side;
    a.Pd = p.Pd;
    a.RW = rows;
    a.tile_stride = pair_tile_stride(es, rows, s.WD);
    a.pbase = p0;
    a.pend = p1;
    a.zoff = b.zoff;
    a.row0 = b.row0;
    a.nsplit = s.nsplit;
    a.wait_ns = p.wait_ns > 0 ? (unsigned long long)p.wait_ns : kWaitLimitNs;
    a.fault = p.test_fault;
    if (direct) {
        a.nviews = p.g.P;
        a.vstep = 1;
        a.scale = (float)(M_PI / (double)p.g.P);
    } else {
        a.nviews = p.Pd;
        a.vstep = p.D;
        a.scale = (float)(M_PI / (double)p.Pd);
    }
    launched = true;
    if (!direct) return launch_pair_od(s, map, a, ss.nsq, st);
    switch (p.qtype) {
        case FDKOD_F32: return launch_pair_f32(s, map, a, ss.nsq, st);
        case FDKOD_BF16: return launch_pair_bf16(s, map, a, ss.nsq, st);
        case FDKOD_F16: return launch_pair_f16(s, map, a, ss.nsq, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_backproject_pairs(const PlanImpl &p, const SquareSet &ss, bool direct, const void *src,
                                     float *vol, cudaStream_t st, int p0, int p1, bool &launched) {
    launched = false;
    PairShape s;
    if (!pair_shape(p, ss, direct, true, (p.g.N + 1) / 2, s)) return cudaSuccess;
    Band whole;
    whole.nrows = p.g.Nv;
    return try_launch_pair(p, ss, direct, src, vol, st, s, whole, p0, p1, launched);
}

int pair_slab(const PlanImpl &p, const SquareSet &ss, bool direct) {
    PairShape s;
    return pair_shape(p, ss, direct, true, (p.g.N + 1) / 2, s) ? s.zp : 16;
}

void backproject_form(const PlanImpl &p, int nz, fdkod_forms &f) {
    const bool direct = p.D == 1, whole = nz == 0 || nz == p.g.N;
    const int es = (direct && p.qtype != FDKOD_F32) ? 2 : 4, pairs = ((whole ? p.g.N : nz) + 1) / 2;
    PairShape s;
    if ((direct && ((size_t)p.g.Nu * es) % 16 != 0) || !pair_shape(p, p.od, direct, whole, pairs, s)) return;
    f.bp_slices = s.zp;
    f.bp_columns = s.WD;
    f.bp_views = s.vps;
    f.bp_slots = s.slots;
    f.bp_split = s.nsplit;
}

cudaError_t launch_backproject(const PlanImpl &p, const SquareSet &ss, bool direct, const void *src, float *vol,
                               cudaStream_t st, Band b) {
    const bool whole = b.row0 == 0 && (b.nrows < 0 || b.nrows == p.g.Nv) && b.zoff == 0 && (b.nz < 0 || b.nz == p.g.N);
    if (b.nrows < 0) b.nrows = p.g.Nv;
    if (b.nz < 0) b.nz = p.g.N;
    bool launched = false;
    PairShape s;
    cudaError_t pe = cudaSuccess;
    if (whole)
        pe = launch_backproject_pairs(p, ss, direct, src, vol, st, 0, (p.g.N + 1) / 2, launched);
    else if (pair_shape(p, ss, direct, false, (b.nz + 1) / 2, s))
        pe = try_launch_pair(p, ss, direct, src, vol, st, s, b, b.zoff, b.zoff + b.nz, launched);
    if (launched || pe != cudaSuccess) return pe;
    BpParams a{};
    a.src = src;
    a.vol = vol;
    a.geo = ss.geo;
    a.crop = ss.crop;
    a.w0 = ss.w0;
    a.status = p.status;
    a.N = p.g.N;
    a.P = p.g.P;
    a.Nv = p.g.Nv;
    a.m = ss.m;
    a.tps = ss.tiles_per_side;
    a.Wd = ss.Wd;
    a.Rw = ss.Rw;
    const size_t per_view = sizeof(float) * (size_t)ss.Rw * (ss.Wd + 1);
    a.J = (int)std::min<size_t>(kViewsPerChunk, (200u * 1024u) / per_view);  // 0: the unstaged kernel
    a.row0 = b.row0;
    a.zoff = b.zoff;
    a.nz = b.nz;
    if (direct) {
        a.sq_stride = 0;
        a.view_stride = (long long)b.nrows * p.g.Nu;
        a.row_stride = p.g.Nu;
        a.src_cols = p.g.Nu;
        a.src_rows = b.nrows;
        a.nviews = p.g.P;
        a.vstep = 1;
        a.scale = (float)(M_PI / (double)p.g.P);
        switch (p.qtype) {
            case FDKOD_F32: return launch_t<float, true>(a, ss.nsq, st);
            case FDKOD_BF16: return launch_t<__nv_bfloat16, true>(a, ss.nsq, st);
            case FDKOD_F16: return launch_t<__half, true>(a, ss.nsq, st);
        }
        return cudaErrorInvalidValue;
    }
    a.view_stride = (long long)b.nrows * p.Tstride;
    a.sq_stride = (long long)p.Pd * a.view_stride;
    a.row_stride = p.Tstride;
    a.src_cols = p.Tstride;
    a.src_rows = b.nrows;
    a.nviews = p.Pd;
    a.vstep = p.D;
    a.scale = (float)(M_PI / (double)p.Pd);
    return launch_t<float, false>(a, ss.nsq, st);
}

// ---- batch of plans, one persistent launch --------------------------------

struct BatchImpl {
    CUtensorMap *maps = nullptr;
    BatchInst *insts = nullptr;
    int4 *items = nullptr;
    int *counter = nullptr;
    int nitems = 0;
    size_t smem = 0;
    int grid = 0;
};

namespace {
void batch_free_impl(BatchImpl *b) {
    cudaFree(b->maps);
    cudaFree(b->insts);
    cudaFree(b->items);
    cudaFree(b->counter);
    delete b;
}
}  // namespace

cudaError_t batch_create(const PlanImpl *const *plans, const void *const *src, float *const *vols, int count,
                         BatchImpl **out, bool &supported) {
    supported = false;
    *out = nullptr;
    std::vector<CUtensorMap> maps((size_t)count);
    std::vector<BatchInst> insts((size_t)count);
    std::vector<std::pair<double, int>> order;
    size_t smem = 0;
    for (int i = 0; i < count; ++i) {
        const PlanImpl &p = *plans[i];
        const bool direct = p.D == 1;
        if (direct && p.qtype != FDKOD_F32) return cudaSuccess;  // 16-bit windows: not in the batch form
        Band b;
        b.nrows = p.g.Nv;
        b.nz = p.g.N;
        int WD = 0;
        if (!make_tma_launch(p, p.od, direct, src[i], vols[i], b, maps[i], insts[i].a, WD)) return cudaSuccess;
        insts[i].direct = direct ? 1 : 0;
        insts[i].WD = WD;
        smem = std::max(smem, sizeof(float) * (size_t)2 * kViewsPerStage * insts[i].a.tile_stride + 128);
        order.push_back({-(double)p.g.N * p.g.N * p.g.N * (double)insts[i].a.nviews, i});
    }
    // two stages of the widest windows must fit a block beside the static shared memory
    cudaFuncAttributes fa{};
    int optin = 0, dev0 = 0;
    cudaError_t ae = cudaFuncGetAttributes(&fa, bp_persistent_kernel);
    if (ae == cudaSuccess) ae = cudaGetDevice(&dev0);
    if (ae == cudaSuccess) ae = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev0);
    if (ae != cudaSuccess) return ae;
    if (smem + fa.sharedSizeBytes > (size_t)optin) return cudaSuccess;
    std::sort(order.begin(), order.end());
    std::vector<int4> items;
    for (const auto &oi : order) {
        const int i = oi.second;
        const BpTmaParams &a = insts[i].a;
        const int tiles = plans[i]->od.nsq * a.tps * a.tps;
        const int zs = (a.nz + kZT - 1) / kZT;
        for (int t = 0; t < tiles; ++t)
            for (int z = 0; z < zs; ++z) items.push_back(make_int4(i, t, z, 0));
    }
    supported = true;
    cudaError_t e = ensure_smem<bp_persistent_kernel>(smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bp_persistent_kernel, kThreads, smem)) !=
        cudaSuccess)
        return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    BatchImpl *b = new BatchImpl;
    b->nitems = (int)items.size();
    b->smem = smem;
    b->grid = std::min(per_sm * sms, std::max(1, b->nitems));
    if ((e = cudaMalloc(&b->maps, sizeof(CUtensorMap) * count)) != cudaSuccess ||
        (e = cudaMalloc(&b->insts, sizeof(BatchInst) * count)) != cudaSuccess ||
        (e = cudaMalloc(&b->items, sizeof(int4) * std::max<size_t>(1, items.size()))) != cudaSuccess ||
        (e = cudaMalloc(&b->counter, sizeof(int))) != cudaSuccess ||
        (e = cudaMemcpy(b->maps, maps.data(), sizeof(CUtensorMap) * count, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(b->insts, insts.data(), sizeof(BatchInst) * count, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(b->items, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice)) !=
            cudaSuccess) {
        batch_free_impl(b);
        return e;
    }
    *out = b;
    return cudaSuccess;
}

cudaError_t batch_launch(const BatchImpl &b, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(b.counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    bp_persistent_kernel<<<b.grid, kThreads, b.smem, st>>>(b.maps, b.insts, b.items, b.nitems, b.counter);
    return cudaGetLastError();
}

void batch_destroy(BatchImpl *b) {
    if (b) batch_free_impl(b);
}

}  // namespace fdkod
