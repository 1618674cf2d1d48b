// The staged backprojection kernel (bp_pair_kernel) and its launch templates;
// each storage type is instantiated in a file of its own (bp_pair_*.cu), so
// that they compile in parallel.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "fdkod_internal.cuh"
#include "tma.cuh"

namespace fdkod {

struct BpPairParams;
struct PairShape;
// one per source: decomposed data, float32 Q, bfloat16 Q, float16 Q
cudaError_t launch_pair_od(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                           cudaStream_t st);
cudaError_t launch_pair_f32(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                            cudaStream_t st);
cudaError_t launch_pair_bf16(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                             cudaStream_t st);
cudaError_t launch_pair_f16(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                            cudaStream_t st);

// Staged backprojection, two slabs of ZP slices per CTA.  A thread owns the
// slices of both slabs in one (x, y) column, as the two lanes of packed FP32
// arithmetic: the column weights and the per-view set-up serve both.
//
// MIRROR (whole volumes): the slices p0 .. p0 + ZP - 1 of the lower half and
// their mirror images N - 1 - p about the mid-plane z = 0.  A voxel and its
// mirror read the same column (Eq. 1 does not involve z) and mirrored rows:
// z/U + (Nv-1)/2 and -z/U + (Nv-1)/2 add up to Nv - 1.  So the row fraction is
// shared too, and with the two windows of a view staged at row origins vlo and
// vlo', the mirror's window row is C - v for C = Nv - 1 - vlo - vlo'.
//
// Otherwise (slabs of a volume, bands of detector rows): 2 ZP consecutive
// slices, the second slab's rows with a coordinate of their own.
//
// What bounds it is instruction issue (a packed two-lane FP32 instruction
// reads its operands over two issue slots) together with the shared-memory
// path.  So slices go in groups that read consecutive rows at compile-time
// offsets from one address (pair_slices): no address, row or fraction
// arithmetic in integers per slice, and each row is loaded and
// column-interpolated once per group, also where 1/U > 1 (before: both rows
// of every such slice).  ncu, 256^3 x 90 views: 28.7 -> 20.3 warp instructions
// and 6.5 -> 4.9 shared loads per slice pair.  A warp covers 8 x 4 columns (16 x 2:
// 5 % bank conflicts, now none).  Backprojection of 512^3 x 180 views:
// 10.80 ms before, 8.61 ms with ZP = 16, 8.25 ms with ZP = 32 (1024^3 x 90
// views 42.9 -> 33.0 ms); a 64-slice slab of 2000^3 from 45 views, not mirrored:
// 6.9 ms before (one voxel at a time, 18.7 instructions each), 5.4 ms.
struct BpPairParams {
    float *vol;
    const GeomEntry *geo;
    const int32_t *crop;
    const int32_t *w0;
    int *status;
    int N, P, Nv, m, tps;
    int nviews, vstep, Pd;
    int RW, tile_stride;  // rows of a ZP-slice window; elements per staged window
    // MIRROR: slice pairs pbase .. pend - 1 (pair p: slices p and N - 1 - p);
    // otherwise slices pbase .. pend - 1, written to vol[z - zoff]
    int pbase, pend, zoff;
    int row0;             // detector row held in the source's row 0
    int nsplit;           // SPLIT: CTAs of a cluster that share the views
    float scale;
    unsigned long long wait_ns;
    int fault;
};

// What a launch needs besides its parameters: the window width, slices per
// slab, views per ring slot, slots and CTAs per cluster pick the instantiation.
struct PairShape {
    int WD, zp, vps, slots, nsplit;
    bool mirror;
};

namespace {

constexpr int kThreads = kTile * kTile;

constexpr uint64_t kWaitLimitNs = 2000000000ull;
// test hooks of the failure paths (fdkod_set_test_fault)
constexpr int kTestFaultSkipCopy = 1;    // CTA 0 leaves out one copy of its chunk 1
constexpr int kTestFaultSmallWindow = 2; // every window counts as too small

__device__ __forceinline__ void square_range(int q, int m, int N, int &i0, int &i1) {
    i0 = (int)(((long long)q * N + m - 1) / m);
    i1 = (int)((((long long)q + 1) * N + m - 1) / m) - 1;
}

// shared-memory load of one window element at a compile-time byte offset
// from a 32-bit address, widened to float32
template <typename TS, int OFF>
struct Lds;
template <int OFF>
struct Lds<float, OFF> {
    static __device__ __forceinline__ float f(uint32_t addr) {
        float v;
        asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(OFF) : "memory");
        return v;
    }
};
template <int OFF>
struct Lds<__nv_bfloat16, OFF> {
    static __device__ __forceinline__ float f(uint32_t addr) {
        uint32_t u;
        asm volatile("ld.shared.u16 %0, [%1+%2];" : "=r"(u) : "r"(addr), "n"(OFF) : "memory");
        return __uint_as_float(u << 16);  // bfloat16 is the top half of a float32
    }
};
template <int OFF>
struct Lds<__half, OFF> {
    static __device__ __forceinline__ float f(uint32_t addr) {
        unsigned short h;
        asm volatile("ld.shared.u16 %0, [%1+%2];" : "=h"(h) : "r"(addr), "n"(OFF) : "memory");
        return __half2float(__ushort_as_half(h));
    }
};

// 1 / x for normal x, to an ulp (one MUFU instruction)
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Barriers over all threads of the cluster (ordering their shared memory) and
// over the consumer warps.  Both take whole warps and have no time limit, so
// each brings its warp together first: callers come from code that diverges
// (one lane hands a slot back, ragged tiles store under a condition).
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int THREADS>
__device__ __forceinline__ void consumers_sync() {
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}
// two floats at this CTA's shared address a, of the cluster's CTA `rank`
__device__ __forceinline__ float2 ld_cluster(uint32_t a, uint32_t rank) {
    float2 v;
    asm volatile("{\n\t.reg .u32 ra;\n\tmapa.shared::cluster.u32 ra, %2, %3;\n\t"
                 "ld.shared::cluster.v2.f32 {%0, %1}, [ra];\n\t}"
                 : "=f"(v.x), "=f"(v.y)
                 : "r"(a), "r"(rank)
                 : "memory");
    return v;
}

// Column-interpolated samples (U^-2 weighted) of row r + K of the first slab's
// window (at aL + K ROWB) and of row r' + K of the second's (aU + K ROWB;
// MIRROR: row C - r - K, at aU - K ROWB).
template <typename TS, uint32_t ROWB, bool MIRROR, int K>
__device__ __forceinline__ float2 pair_row(uint32_t aL, uint32_t aU, float2 A0, float2 A1) {
    constexpr int ES = (int)sizeof(TS);
    constexpr int OL = K * (int)ROWB, OU = MIRROR ? -OL : OL;
    return __ffma2_rn(A1, make_float2(Lds<TS, OL + ES>::f(aL), Lds<TS, OU + ES>::f(aU)),
                      __fmul2_rn(A0, make_float2(Lds<TS, OL>::f(aL), Lds<TS, OU>::f(aU))));
}

// One slice of a group: with t in [-1, 1) the row coordinate relative to the
// middle one of three consecutive rows c0, c1, c2, the row interpolation is
// (1 - |t|) c1 + |t| (t < 0 ? c0 : c2): no row but the two around the sample
// enters it.  t.y: the second slab's coordinate (MIRROR: unused, t.x serves
// both).  t runs as scalar sums: a packed add measured 3 % slower.
template <typename TS, uint32_t ROWB, bool MIRROR, int G, int I>
__device__ __forceinline__ void pair_group(float2 *acc, float2 c0, float2 c1, float2 t, float du, uint32_t aL,
                                           uint32_t aU, float2 A0, float2 A1) {
    if constexpr (I < G) {
        const float2 c2 = pair_row<TS, ROWB, MIRROR, I + 2>(aL, aU, A0, A1);
        if constexpr (MIRROR) t.y = t.x;
        const bool lo = t.x < 0.f, lo2 = MIRROR ? lo : t.y < 0.f;
        const float2 y = make_float2(lo ? -c0.x : c2.x, lo2 ? -c0.y : c2.y);
        const float w1 = 1.0f - fabsf(t.x), w2 = MIRROR ? w1 : 1.0f - fabsf(t.y);
        acc[I] = __ffma2_rn(t, y, __ffma2_rn(make_float2(w1, w2), c1, acc[I]));
        pair_group<TS, ROWB, MIRROR, G, I + 1>(acc, c1, c2, make_float2(t.x + du, MIRROR ? 0.f : t.y + du), du, aL, aU,
                                               A0, A1);
    }
}

// floor of |x| < 2^22 through the float 1.5 2^23 + floor(x) (unit spacing,
// rounded down): its bits are kFloorBits + floor(x), so an address takes one
// multiply-add, and no conversion instruction is needed
constexpr float kFloorBias = 12582912.0f;  // 1.5 * 2^23
constexpr uint32_t kFloorBits = 0x4B400000u;
__device__ __forceinline__ float floor_biased(float x) { return __fadd_rd(x, kFloorBias); }

// The ZP slice pairs of one column in groups of G consecutive ones, for a
// drift |1/U - 1| of at most 1 / (G - 1) rows per slice: then slice g + i of
// a group reads two of the rows b + i, b + i + 1, b + i + 2 for one b, so a
// group loads G + 2 rows at compile-time offsets from one address.  w is the
// window row of the slab's centre less the centre's slice number: a number of
// a few rows whatever ZP, so its rounding stays below a row coordinate's (w2:
// the second slab's; MIRROR: unused, bU is then KU).
template <typename TS, uint32_t ROWB, bool MIRROR, int G, int ZP>
__device__ __forceinline__ void pair_slices(float2 (&acc)[ZP], float w, float w2, float du, uint32_t bL, uint32_t bU,
                                            float2 A0, float2 A1) {
#pragma unroll
    for (int g = 0; g < ZP; g += G) {
        // window row less slice number at the group's ends -> its first row's
        // address and the first slice's coordinate relative to the row after it
        constexpr float kMid = 0.5f * (float)(ZP - 1);
        auto start = [&](float wc, uint32_t base, float &t0) -> uint32_t {
            const float first = fmaf((float)g - kMid, du, wc), last = fmaf((float)(g + G - 1) - kMid, du, wc);
            const float bm = floor_biased(fminf(first, last));
            t0 = first - (bm - (kFloorBias - 1.0f));  // first - (b + 1), exact
            return __float_as_uint(bm) * ROWB + (base + ((uint32_t)g - kFloorBits) * ROWB);
        };
        float2 t0;
        const uint32_t aL = start(w, bL, t0.x);
        uint32_t aU;
        if constexpr (MIRROR) aU = bU - aL;
        else aU = start(w2, bU, t0.y);
        pair_group<TS, ROWB, MIRROR, G, 0>(acc + g, pair_row<TS, ROWB, MIRROR, 0>(aL, aU, A0, A1),
                                           pair_row<TS, ROWB, MIRROR, 1>(aL, aU, A0, A1), t0, du, aL, aU, A0, A1);
    }
}

// Any 1/U: both rows of every slice at an address of its own.  Row
// coordinates in 9.23 fixed point: the row is V >> 23, the fraction's float
// is V's mantissa bits under the exponent of 1.0.
template <typename TS, uint32_t ROWB, bool MIRROR, int ZP>
__device__ __forceinline__ void pair_slices_any(float2 (&acc)[ZP], float w, float w2, float invU, uint32_t bL,
                                                uint32_t bU, float2 A0, float2 A1) {
    constexpr float kFix = 8388608.0f;  // 2^23
    auto fixed = [&](float wc) { return __float2uint_rn(fmaf(-0.5f * (float)(ZP - 1), invU - 1.0f, wc) * kFix); };
    uint32_t V = fixed(w), V2 = MIRROR ? 0u : fixed(w2);
    const uint32_t dV = __float2uint_rn(invU * kFix);
#pragma unroll
    for (int i = 0; i < ZP; ++i) {
        const uint32_t aL = (V >> 23) * ROWB + bL, aU = MIRROR ? bU - aL : (V2 >> 23) * ROWB + bU;
        const float2 A = pair_row<TS, ROWB, MIRROR, 0>(aL, aU, A0, A1), B = pair_row<TS, ROWB, MIRROR, 1>(aL, aU, A0, A1);
        // fb = 1 + f exactly, so 1 - f and f are exact
        const float fb = __uint_as_float((V & 0x7fffffu) | 0x3f800000u);
        const float fb2 = MIRROR ? fb : __uint_as_float((V2 & 0x7fffffu) | 0x3f800000u);
        acc[i] = __ffma2_rn(make_float2(fb - 1.0f, fb2 - 1.0f), B,
                            __ffma2_rn(make_float2(2.0f - fb, 2.0f - fb2), A, acc[i]));
        V += dV;
        if constexpr (!MIRROR) V2 += dV;
    }
}

// Warp-specialised: warp 8 is the producer (per chunk of VPS views it finds
// the windows, writes the view parameters and issues the copies into a ring
// of SLOTS slots); warps 0-7 consume.  A slot is full when its copies
// have landed (full[slot], which also publishes the producer's parameters)
// and free again when the consumer warps have arrived on empty[slot]:
// no block-wide barrier inside the view loop, so consumer warps drift within
// the ring instead of waiting for the slowest.  Every wait is bounded
// (FDKOD_ERR_TIMEOUT); a producer that gives up waits for its copies in
// flight before it leaves.  The producer polls `empty` (mbarrier.test_wait):
// suspended in mbarrier.try_wait it was measured to resume late (the whole
// kernel 1.4x slower); the consumers' waits on `full` are mostly satisfied
// at once and suspend (polling them measured no faster).
struct PairView {
    float4 a;   // cos, sin, 1/d_c, alpha
    float4 b;   // gamma, g, column offset, window row of the first slab's centre less its slice number
    float zcr;  // z_c / d_c (first slab)
    int group;  // slices per group (pair_slices), 0: any drift, -1: window too small, skip the view
    // byte addresses of row 0, column -kFloorBits of the first window, and of
    // the second one; MIRROR: of the second's row C plus the former (row r of
    // the first window at aL = baseL + r ROWB + ..., row C - r of the second
    // one at baseU - aL)
    uint32_t baseL, baseU;
    float w2, zcr2;  // second slab: as b.w and zcr (not MIRROR)
    float pad[2];
};
// a group's first or last row may lie one row outside its window (such a row
// never enters a sum): one row of the widest window before and after the ring
constexpr int kPairPad = 512;
constexpr int kPairViews = 2;                      // views per slot, at most (16 producer lanes each)
constexpr int kPairConsumers = kThreads / 32;      // 8
constexpr int kPairThreads = kThreads + 32;        // plus the producer warp
// CTAs per SM: registers decide (2 ZP accumulators per thread)
constexpr int pair_ctas(int ZP) { return ZP == 32 ? 2 : 3; }

// SPLIT: the nsplit CTAs of a cluster (grid z) take a range of the views each
// and add up their sums through distributed shared memory, CTA r every
// nsplit-th slice from r on, in the order of the ranges (pair_shape says where).
template <typename TS, bool DIRECT, bool MIRROR, int WD, int ZP, int VPS, int SLOTS, bool SPLIT>
__global__ void __launch_bounds__(kPairThreads, pair_ctas(ZP))
bp_pair_kernel(const __grid_constant__ CUtensorMap tmap, BpPairParams a) {
    constexpr int ES = (int)sizeof(TS);
    constexpr int kAl = 16 / ES;
    constexpr uint32_t ROWB = (uint32_t)(ES * WD);  // bytes per window row
    static_assert(VPS <= kPairViews, "the producer warp sets up a view on 16 lanes");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    TS *sm = (TS *)(smem_raw + ((128u - (tma::smem_u32(smem_raw) & 127u)) & 127u) + kPairPad);
    const uint32_t sbase = tma::smem_u32(sm);
    __shared__ __align__(8) uint64_t full[SLOTS], empty[SLOTS];
    __shared__ PairView s_view[SLOTS * VPS];

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
    const int p0 = a.pbase + blockIdx.y * (MIRROR ? ZP : 2 * ZP);  // first slice (pair)

    const float half_n = 0.5f * (float)(a.N - 1);
    const float xc = 0.5f * ((float)ix0 + (float)ix1) - half_n;
    const float yc = 0.5f * ((float)iy0 + (float)iy1) - half_n;
    // centres of the slabs (a second slab wholly past the end repeats the
    // first one: a slab may run past the volume, but not start there)
    const float zc = (float)p0 + 0.5f * (float)(ZP - 1) - half_n;
    const float zc2 = MIRROR ? -zc : (p0 + ZP < a.pend ? zc + (float)ZP : zc);
    const float vcd = 0.5f * (float)(a.Nv - 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's views
    const int j0 = SPLIT ? a.nviews * (int)blockIdx.z / a.nsplit : 0;
    const int nviews = SPLIT ? a.nviews * ((int)blockIdx.z + 1) / a.nsplit - j0 : a.nviews;
    const int nch = (nviews + VPS - 1) / VPS;
    // window of view w of slot sl, first (h = 0) or second (h = 1) slab
    auto win = [&](int sl, int w, int h) { return (uint32_t)((sl * VPS + w) * 2 + h) * (uint32_t)a.tile_stride; };

    if (threadIdx.x == 0) {
        // warps with a column of the tile (8 x 4 each); the others leave at once
        // unless MIRROR
        const int busy = ((xe - x0) / 8 + 1) * ((ye - y0) / 4 + 1);
        for (int i = 0; i < SLOTS; ++i) {
            tma::mbar_init(&full[i], 1);
            tma::mbar_init(&empty[i], MIRROR ? kPairConsumers : busy);
        }
        tma::fence_mbar_init();
    }
    __syncthreads();

    if (warp == kPairConsumers) {
        // ---- producer: lanes 16 w .. 16 w + 15 set up view w of the chunk,
        // 0-7 of them at the corners of the first slab, 8-15 of the second
        const int32_t w0q = a.w0[q];
        const int w = lane >> 4, cc = lane & 7;
        const float zcl = (lane & 8) ? zc2 : zc;
        const float cx = (float)((cc & 1) ? xe : x0) - half_n - xc;
        const float cy = (float)((cc & 2) ? ye : y0) - half_n - yc;
        const float cz = (cc & 4) ? 0.5f * (float)(ZP - 1) : -0.5f * (float)(ZP - 1);
        int c = 0;
        for (; c < nch; ++c) {
            const int sl = c % SLOTS;
            const int nj = min(VPS, nviews - c * VPS);
            const int j = j0 + c * VPS + min(w, nj - 1);  // lanes past the chunk repeat its last view
            const int k = j * a.vstep;
            const size_t o = (size_t)q * a.P + k;
            const GeomEntry ge = a.geo[o];
            const int cbase = DIRECT ? a.crop[o] : 0;
            const float toff = DIRECT ? ge.frac - (float)w0q : -(float)w0q;
            const float dd = fmaf(ge.cb, cx, ge.sb * cy);
            const float invU = __fdividef(ge.g_hi, fmaf(ge.r, dd, 1.0f));
            const float t = fmaf(invU, fmaf(ge.alpha, cx, ge.gamma * cy), toff);
            const float zcr = zcl * ge.r;
            // z_c g as hi + lo (exact product error by FMA)
            const float ph = zcl * ge.g_hi;
            const float pl = fmaf(zcl, ge.g_lo, fmaf(zcl, ge.g_hi, -ph));
            const float v = (ph + vcd) + (pl + invU * (cz - zcr * dd));
            float tmin = t, tmax = t, vmin = v, vmax = v;
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) {  // within each half's 8 corners
                vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, off));
                vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, off));
            }
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) {  // columns: both halves
                tmin = fminf(tmin, __shfl_xor_sync(0xffffffffu, tmin, off));
                tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, off));
            }
            const float vmin2 = __shfl_down_sync(0xffffffffu, vmin, 8);
            const float vmax2 = __shfl_down_sync(0xffffffffu, vmax, 8);
            // lane 16 w: columns read floor(t) .. floor(t) + 1 over the tile,
            // one sample of slack each side for FP32 rounding
            const int clo = cbase + (int)floorf(tmin) - 1;
            const int chi = cbase + (int)floorf(tmax) + 2;
            const int xs = clo & ~(kAl - 1);  // 16-byte aligned start of the copy
            const int vlo = (int)floorf(vmin) - 1, vhi = (int)floorf(vmax) + 2;
            const int vlo2 = (int)floorf(vmin2) - 1, vhi2 = (int)floorf(vmax2) + 2;
            // largest drift per slice over the tile (1/U is monotone in x
            // and y), with a margin for rounding
            float drift = fabsf(invU - 1.0f);
#pragma unroll
            for (int off = 2; off > 0; off >>= 1) drift = fmaxf(drift, __shfl_xor_sync(0xffffffffu, drift, off));
            // round r of a slot may start once its round r - 1 was consumed
            // (lane 0 waits; the warp follows its answer)
            bool ok = true;
            if (c >= SLOTS && lane == 0)
                ok = tma::mbar_wait_spin(&empty[sl], (uint32_t)(((c / SLOTS) & 1) ^ 1), a.wait_ns);
            if (!__shfl_sync(0xffffffffu, ok, 0)) {
                if (lane == 0) atomicOr(a.status, 2);
                break;
            }
            // the row coordinate of a slab's centre, less its slice number
            const float wcen = (ph - ((float)vlo - vcd + 0.5f * (float)(ZP - 1))) + pl;
            if (!MIRROR && (lane & 15) == 8 && w < nj) {
                s_view[sl * VPS + w].w2 = wcen;
                s_view[sl * VPS + w].zcr2 = zcr;
            }
            const bool lead = (lane & 15) == 0 && w < nj;
            if (lead) {
                const bool skip = (chi - xs > WD - 1) || (vhi - vlo > a.RW - 1) || (vhi2 - vlo2 > a.RW - 1) ||
                                  a.fault == kTestFaultSmallWindow;
                if (skip) atomicOr(a.status, 1);
                PairView &pv = s_view[sl * VPS + w];
                pv.a = make_float4(ge.cb, ge.sb, ge.r, ge.alpha);
                pv.b = make_float4(ge.gamma, ge.g_hi, toff - (float)(xs - cbase), wcen);
                pv.zcr = zcr;
                pv.group = skip ? -1
                           : drift * 15.f < 0.999f ? 16
                           : drift * 7.f < 0.999f  ? 8
                           : drift * 3.f < 0.999f  ? 4
                                                   : 0;
                const uint32_t bL = sbase + (uint32_t)ES * (win(sl, w, 0) - kFloorBits);
                const uint32_t bU = sbase + (uint32_t)ES * (win(sl, w, 1) - kFloorBits);
                pv.baseL = bL;
                pv.baseU = MIRROR ? (uint32_t)((a.Nv - 1) - vlo - vlo2) * ROWB + bU + bL : bU;
            }
            // the copies: lane 0 for every view of the chunk
            const int xs0 = __shfl_sync(0xffffffffu, xs, 0), xs1 = __shfl_sync(0xffffffffu, xs, 16);
            const int vl0 = __shfl_sync(0xffffffffu, vlo, 0), vl1 = __shfl_sync(0xffffffffu, vlo, 16);
            const int vu0 = __shfl_sync(0xffffffffu, vlo2, 0), vu1 = __shfl_sync(0xffffffffu, vlo2, 16);
            const int tz = DIRECT ? k : q * a.Pd + j;
            const int tz0 = __shfl_sync(0xffffffffu, tz, 0), tz1 = __shfl_sync(0xffffffffu, tz, 16);
            __syncwarp();  // the parameters are written before lane 0 publishes them
            if (lane == 0) {
                tma::fence_proxy_async();
                tma::mbar_arrive_expect_tx(&full[sl], (uint32_t)(nj * 2 * a.RW * WD * ES));
                for (int v2 = 0; v2 < nj; ++v2) {
                    // test hook: the slot's bytes never all arrive, its wait runs out
                    if (a.fault == kTestFaultSkipCopy && c == 1 && v2 == 0 && blockIdx.x + blockIdx.y + blockIdx.z == 0)
                        continue;
                    const int x = v2 == 0 ? xs0 : xs1, z = v2 == 0 ? tz0 : tz1;
                    // rows of the source (out of range: zero fill)
                    tma::load_3d(sm + win(sl, v2, 0), &tmap, &full[sl], x, (v2 == 0 ? vl0 : vl1) - a.row0, z);
                    tma::load_3d(sm + win(sl, v2, 1), &tmap, &full[sl], x, (v2 == 0 ? vu0 : vu1) - a.row0, z);
                }
            }
            __syncwarp();
        }
        // copies still in flight must land before the CTA may exit
        if (lane == 0)
            for (int m = max(0, c - SLOTS); m < c; ++m)
                tma::mbar_wait_bounded(&full[m % SLOTS], (uint32_t)((m / SLOTS) & 1), a.wait_ns);
        if constexpr (SPLIT) {
            cluster_sync();
            cluster_sync();
        }
        return;
    }

    // ---- consumers.  The voxels of the two slabs go through the same
    // operations on different samples, so they share packed two-lane FP32
    // instructions (x: first slab, y: second; each lane rounds as the scalar
    // operation would).
    const int x = x0 + (warp & 1) * 8 + (lane & 7), y = y0 + (warp >> 1) * 4 + (lane >> 3);
    const bool active = x <= xe && y <= ye;
    // threads outside a ragged tile repeat its last column (inside the
    // window) and store nothing
    const float dx = (float)min(x, xe) - half_n - xc, dy = (float)min(y, ye) - half_n - yc;
    float2 acc[ZP];  // (first slab, second slab)
#pragma unroll
    for (int i = 0; i < ZP; ++i) acc[i] = make_float2(0.f, 0.f);

    // A warp wholly outside a ragged tile takes no part: its work would take issue
    // slots from the others (367^3, squares of 23 voxels: 4.30 -> 3.21 ms; 306^3 x 428
    // bf16, squares of 38, D = 1: 8.41 -> 7.02 ms).  Not mirrored, it leaves (`empty`
    // does not count it); mirrored, it hands the slots back.  How it is asked
    // moves the registers of the view loop: mirrored, this vote inside the loop
    // saves spills (512^3 8.35 -> 8.25 ms; 8.34 by the tile's extent); otherwise the
    // extent (a 64-slice slab of 2000^3 with its decomposition 10.40 -> 10.38 ms; 10.53
    // by the vote, 10.43 with a loop that hands the slots back).
    const bool idle = MIRROR ? !__any_sync(0xffffffffu, active)
                             : (warp & 1) * 8 > xe - x0 || (warp >> 1) * 4 > ye - y0;
    if (!MIRROR && idle) return;
    const int mine = MIRROR && idle ? 0 : VPS;
    int sl = 0, left = nviews;
    uint32_t phase = 0;
    for (; left > 0; left -= VPS) {
        const bool ok = tma::mbar_wait_bounded(&full[sl], phase, a.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicOr(a.status, 2);
            if constexpr (SPLIT) break;  // the cluster's barriers wait for this warp
            return;                      // the producer waits for the copies in flight
        }
        const PairView *pv = s_view + sl * VPS, *pe = pv + min(mine, left);
#pragma unroll 1
        for (; pv != pe; ++pv) {
            const int group = pv->group;  // uniform per CTA
            const float4 pa = pv->a;
            const float4 pb = pv->b;
            const float dd = fmaf(pa.x, dx, pa.y * dy);
            // one Newton step on the reciprocal: its error scales with the
            // distance from the slab's centre, which 32 pairs double
            const float den = fmaf(pa.z, dd, 1.0f), r0 = rcp_approx(den);
            const float invU = pb.y * fmaf(r0, fmaf(-den, r0, 1.0f), r0);
            const float du = invU - 1.0f;
            const float t = fmaf(invU, fmaf(pa.w, dx, pb.x * dy), pb.z);
            const float tm = floor_biased(t);
            const float wgt = invU * invU;
            const float a1 = wgt * (t - (tm - kFloorBias));
            const float a0 = wgt - a1;
            const float2 A1 = make_float2(a1, a1), A0 = make_float2(a0, a0);
            // window rows of the column at the slabs' centres, less the
            // centres' slice numbers
            const float wc = fmaf(-invU, pv->zcr * dd, pb.w);
            const float wc2 = MIRROR ? 0.f : fmaf(-invU, pv->zcr2 * dd, pv->w2);
            const uint32_t col = (uint32_t)ES * __float_as_uint(tm);
            const uint32_t bL = pv->baseL + col, bU = pv->baseU + (MIRROR ? 2u : 1u) * col;
            if (group == 16) {
                pair_slices<TS, ROWB, MIRROR, 16, ZP>(acc, wc, wc2, du, bL, bU, A0, A1);
            } else if (group == 8) {
                pair_slices<TS, ROWB, MIRROR, 8, ZP>(acc, wc, wc2, du, bL, bU, A0, A1);
            } else if (group == 4) {
                pair_slices<TS, ROWB, MIRROR, 4, ZP>(acc, wc, wc2, du, bL, bU, A0, A1);
            } else if (group == 0) {
                pair_slices_any<TS, ROWB, MIRROR, ZP>(acc, wc, wc2, invU, bL, bU, A0, A1);
            }
        }
        __syncwarp();
        if (lane == 0) tma::mbar_arrive(&empty[sl]);  // this warp is done with the slot
        if (++sl == SLOTS) {
            sl = 0;
            phase ^= 1u;
        }
    }
    if constexpr (SPLIT) {
        // every warp is done with the ring: it takes this CTA's sums [i][thread]
        consumers_sync<32 * kPairConsumers>();
        float2 *part = (float2 *)sm + threadIdx.x;
#pragma unroll
        for (int i = 0; i < ZP; ++i) part[i * 32 * kPairConsumers] = acc[i];
        cluster_sync();
        for (int i = (int)blockIdx.z; i < ZP; i += a.nsplit) {
            float2 sum = make_float2(0.f, 0.f);
            for (int r = 0; r < a.nsplit; ++r)
                sum = __fadd2_rn(sum, ld_cluster(tma::smem_u32(part + i * 32 * kPairConsumers), (uint32_t)r));
            const int pz = p0 + i;
            if (active && pz < a.pend) {
                static_assert(!SPLIT || MIRROR, "whole volumes only");
                const int zu = a.N - 1 - pz;
                a.vol[((size_t)pz * a.N + y) * a.N + x] = sum.x * a.scale;
                if (zu != pz) a.vol[((size_t)zu * a.N + y) * a.N + x] = sum.y * a.scale;
            }
        }
        cluster_sync();  // the others may still be reading this CTA's sums
        return;
    }
    if (active) {
#pragma unroll
        for (int i = 0; i < ZP; ++i) {
            const int pz = p0 + i;
            if constexpr (MIRROR) {
                if (pz < a.pend) {
                    const int zu = a.N - 1 - pz;
                    a.vol[((size_t)pz * a.N + y) * a.N + x] = acc[i].x * a.scale;
                    if (zu != pz) a.vol[((size_t)zu * a.N + y) * a.N + x] = acc[i].y * a.scale;
                }
            } else {
                if (pz < a.pend) a.vol[((size_t)(pz - a.zoff) * a.N + y) * a.N + x] = acc[i].x * a.scale;
                if (pz + ZP < a.pend) a.vol[((size_t)(pz + ZP - a.zoff) * a.N + y) * a.N + x] = acc[i].y * a.scale;
            }
        }
    }
}

// elements per staged window of the pair kernel, a 128-byte multiple
inline int pair_tile_stride(int es, int rows, int WD) { return (rows * WD + (128 / es - 1)) & ~(128 / es - 1); }

// dynamic shared memory of the pair kernel: `slots` slots of vps views, two
// windows per view, plus the pads and the 128-byte alignment slack
inline size_t pair_smem(int es, int vps, int slots, int tile_stride) {
    return (size_t)es * slots * vps * 2 * tile_stride + 2 * kPairPad + 128;
}

template <typename TS, bool DIRECT, bool MIRROR, int WD, int ZP, int VPS, int SLOTS, bool SPLIT = false>
cudaError_t launch_pair_t(const CUtensorMap &map, const BpPairParams &prm, int nsq, cudaStream_t st) {
    size_t smem = pair_smem((int)sizeof(TS), VPS, SLOTS, prm.tile_stride);
    // SPLIT: the ring also holds the CTA's sums
    if (SPLIT) smem = std::max(smem, sizeof(float2) * ZP * 32 * kPairConsumers + 2 * (size_t)kPairPad + 128);
    cudaError_t e = ensure_smem<bp_pair_kernel<TS, DIRECT, MIRROR, WD, ZP, VPS, SLOTS, SPLIT>>(smem);
    if (e != cudaSuccess) return e;
    constexpr int kSlices = MIRROR ? ZP : 2 * ZP;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nsq * prm.tps * prm.tps), (unsigned)((prm.pend - prm.pbase + kSlices - 1) / kSlices),
                       SPLIT ? (unsigned)prm.nsplit : 1u);
    cfg.blockDim = dim3(kPairThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = at.val.clusterDim.y = 1;
    at.val.clusterDim.z = SPLIT ? (unsigned)prm.nsplit : 1u;
    cfg.attrs = &at;
    cfg.numAttrs = SPLIT ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, bp_pair_kernel<TS, DIRECT, MIRROR, WD, ZP, VPS, SLOTS, SPLIT>, map, prm);
}

// the shapes pair_shape gives: 32 slices per slab with 2 views per slot and no
// split, a split with whole volumes; 3 slots of 2 views, 2 of 2 or 3 of 1
template <typename TS, bool DIRECT, bool MIRROR, int WD, int ZP, bool SPLIT = false>
cudaError_t launch_pair_v(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                          cudaStream_t st) {
    if (s.vps == 2 && s.slots == 3) return launch_pair_t<TS, DIRECT, MIRROR, WD, ZP, 2, 3, SPLIT>(map, prm, nsq, st);
    if (s.vps == 2) return launch_pair_t<TS, DIRECT, MIRROR, WD, ZP, 2, 2, SPLIT>(map, prm, nsq, st);
    if constexpr (ZP == 16) return launch_pair_t<TS, DIRECT, MIRROR, WD, ZP, 1, 3, SPLIT>(map, prm, nsq, st);
    return cudaErrorInvalidValue;
}

template <typename TS, bool DIRECT, bool MIRROR, int WD>
cudaError_t launch_pair_z(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                          cudaStream_t st) {
    if (s.zp == 32) return launch_pair_v<TS, DIRECT, MIRROR, WD, 32>(s, map, prm, nsq, st);
    if constexpr (MIRROR)
        if (s.nsplit > 1) return launch_pair_v<TS, DIRECT, MIRROR, WD, 16, true>(s, map, prm, nsq, st);
    return launch_pair_v<TS, DIRECT, MIRROR, WD, 16>(s, map, prm, nsq, st);
}

template <typename TS, bool DIRECT, bool MIRROR>
cudaError_t launch_pair_m(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                          cudaStream_t st) {
    switch (s.WD) {
        case 32: return launch_pair_z<TS, DIRECT, MIRROR, 32>(s, map, prm, nsq, st);
        case 48: return launch_pair_z<TS, DIRECT, MIRROR, 48>(s, map, prm, nsq, st);
        case 64: return launch_pair_z<TS, DIRECT, MIRROR, 64>(s, map, prm, nsq, st);
        case 96: return launch_pair_z<TS, DIRECT, MIRROR, 96>(s, map, prm, nsq, st);
        case 128: return launch_pair_z<TS, DIRECT, MIRROR, 128>(s, map, prm, nsq, st);
    }
    return cudaErrorInvalidValue;
}

template <typename TS, bool DIRECT>
cudaError_t launch_pair(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                        cudaStream_t st) {
    return s.mirror ? launch_pair_m<TS, DIRECT, true>(s, map, prm, nsq, st)
                    : launch_pair_m<TS, DIRECT, false>(s, map, prm, nsq, st);
}

}  // namespace
}  // namespace fdkod
