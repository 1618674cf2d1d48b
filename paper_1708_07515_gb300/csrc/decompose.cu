// Decomposition stage of FDK-OD (Sec. 2.1): for every square q, detector row
// v and shifted column t, shift each view's row so the square centre sits
// on one column (linear interpolation at column phi_k + w0 + t, i.e. crop
// column c_qk + t with sub-pixel part f_qk), low-pass it along the view
// axis with symmetric taps h[|i|], |i| < H D (circular over the orbit; the
// triangle (D - |i|) / D^2 with H = 1 by default, a windowed sinc with
// H = 2 as an option) and keep every D-th view.  The views are streamed in
// order: view k = jD + r adds w[r][m] = h[|r + (H - 1 - m) D|] of its sample
// to decimated view j - H + 1 + m, m < 2H, so only 2H running sums are live
// (two for the triangle: (D - r) / D^2 to view j, r / D^2 to view j + 1).
// The stream starts H D - 1 views before view 0 and runs (H - 1) D views
// past the last one (both wrapped): every decimated view sees its whole
// support.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "fdkod_internal.cuh"
#include "tma.cuh"

namespace fdkod {
namespace {

__device__ __forceinline__ float ld_q(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ld_q(const __nv_bfloat16 *p) { return __bfloat162float(__ldg(p)); }
__device__ __forceinline__ float ld_q(const __half *p) { return __half2float(__ldg(p)); }

// floor(a / b) for b > 0
__host__ __device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// Generic path: a warp takes 32 consecutive columns of kGenRows rows, straight
// from global memory (each view's crop row is one run).  The rows share the
// view's crop, shift and weights and keep their loads in flight together; the
// next view's entries are read while this one's samples arrive.  Bound by the
// two loads per sample.  Against one row per thread: 963^3 x 64 rows x 360 views
// f16 1233 -> 688 us, 501^3 x 720 bf16 5.5 -> 3.7 ms (2 rows: 752, 3.7; 8: 749,
// 3.9).  It also beat staging the crops by 4-byte asynchronous copies (501^3
// f32 3.4 against 3.8 ms, 250^3 210 against 255 us).
constexpr int kGenRows = 4, kGenWarps = 8;
template <typename TQ, int H>
__global__ void __launch_bounds__(32 * kGenWarps)
decompose_kernel(const TQ *__restrict__ Q, float *__restrict__ Sp, const int32_t *__restrict__ crop,
                 const GeomEntry *__restrict__ geo, const int32_t *__restrict__ Tq, const float4 *__restrict__ tapw,
                 int Tstride, int P, int D, int Pd, int Nv, int Nu, int rowoff, int rowend, int tiles, int jrange) {
    // grid x: 32-column tiles of every range of decimated views j0 .. j1 - 1
    const int range = blockIdx.x / tiles, j0 = range * jrange, j1 = min(j0 + jrange, Pd);
    const int t = (blockIdx.x - range * tiles) * 32 + threadIdx.x;
    const int v = rowoff + (blockIdx.y * kGenWarps + threadIdx.y) * kGenRows;
    const int q = blockIdx.z;
    if (t >= Tstride || v >= rowend) return;
    const size_t vstride = (size_t)Nv * Tstride;
    float *out = Sp + ((size_t)q * Pd * Nv + v) * Tstride + t;
    const int rows = min(kGenRows, rowend - v);
    if (t >= Tq[q]) {
        for (int j = j0; j < j1; ++j)
            for (int r = 0; r < rows; ++r) out[(size_t)j * vstride + (size_t)r * Tstride] = 0.f;
        return;
    }
    const int32_t *cq = crop + (size_t)q * P;
    const GeomEntry *gq = geo + (size_t)q * P;
    const size_t view = (size_t)Nv * Nu;
    const TQ *Qv = Q + (size_t)v * Nu;
    float acc[kGenRows][2 * H];
#pragma unroll
    for (int r = 0; r < kGenRows; ++r)
#pragma unroll
        for (int m = 0; m < 2 * H; ++m) acc[r][m] = 0.f;
    // block by block from the second view of block j0 - H (its end completes
    // decimated view j0 + 1 - 2 H), the views taken mod P
    int kk = (((j0 - H) * D + 1) % P + P) % P, r0 = 1;
    int c = __ldg(cq + kk) + t;
    float f = __ldg(&gq[kk].frac);
    for (int jst = j0 + 1 - 2 * H; jst < j1; ++jst, r0 = 0) {
        for (int rr = r0; rr < D; ++rr) {
            const TQ *row = Qv + (size_t)kk * view + c;
            const bool in0 = c >= 0 && c < Nu, in1 = c >= -1 && c < Nu - 1;
            float a[kGenRows], b[kGenRows];
#pragma unroll
            for (int r = 0; r < kGenRows; ++r) {
                a[r] = in0 && r < rows ? ld_q(row + r * Nu) : 0.f;
                b[r] = in1 && r < rows ? ld_q(row + r * Nu + 1) : 0.f;
            }
            const float fk = f;
            const float4 w = __ldg(tapw + rr);
            if (++kk == P) kk = 0;
            c = __ldg(cq + kk) + t;
            f = __ldg(&gq[kk].frac);
            const float wm[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int r = 0; r < kGenRows; ++r) {
                const float smp = fmaf(fk, b[r] - a[r], a[r]);
#pragma unroll
                for (int m = 0; m < 2 * H; ++m) acc[r][m] = fmaf(wm[m], smp, acc[r][m]);
            }
        }
        if (jst >= j0)
#pragma unroll
            for (int r = 0; r < kGenRows; ++r)
                if (r < rows) out[(size_t)jst * vstride + (size_t)r * Tstride] = acc[r][0];
#pragma unroll
        for (int r = 0; r < kGenRows; ++r) {
#pragma unroll
            for (int m = 0; m < 2 * H - 1; ++m) acc[r][m] = acc[r][m + 1];
            acc[r][2 * H - 1] = 0.f;
        }
    }
}

// ---------------------------------------------------------------------------
// Staged path: one CTA per (square q, band of detector rows, range of decimated
// views), warp specialised.  The producer warp's lane 0 brings each view's
// crop box (the band's rows x Wc columns from the 16-byte aligned column
// below crop[q][k]) into a ring of slots of kG views with 3D bulk-tensor copies
// (zero fill outside the detector); slot n is full when its bytes have landed
// (mbarrier full[n]) and free again when all consumer warps have arrived on
// empty[n].  No block-wide barrier inside the view loop.
//
// Consumers: lane = detector row, and each warp owns kCW consecutive shifted
// columns of its 32 rows, so a sample is loaded once and serves as the right
// neighbour of one column and the left one of the next: kCW + 1 samples per
// kCW columns, in aligned 16-byte loads.  The box's rows are an odd number
// of 16-byte units long, which keeps those loads free of bank conflicts; the
// crop's offset inside its aligned box is the same for all rows, so it picks
// one of the unrolled bodies (a uniform branch).  Per view and lane: 5 (16-bit
// Q: 3) loads, kCW lerps and kCW 2H tap FMAs.  A view's table entry is loaded
// before the wait for its box (1-2 % faster than after it).  A finished decimated
// view goes through a per-warp transpose buffer, so that its rows leave in
// 64-byte runs, at a pointer that advances by one view per block (computed from
// the view's number: 1 % slower at 512^3 f32, 3 % at 1024^3 bf16, 6 % with 2D taps).
//
// What bounds it: instruction issue for 16-bit Q and 2D-tap filters; for float32
// and the triangle the copies of the crops (~14 |Q| from L2) come close behind:
// ring and copies alone take 0.90 ms of 1.08 at 512^3.  The form before had
// lanes along the columns: two scalar loads per sample, and columns in steps of
// 32 lanes (128 computed for ~100 used).  512^3 x 720 f32: 1.43 -> 1.08 ms with
// the triangle, 2.30 -> 1.475 ms with 2D-tap filters; 1024^3 x 720 bf16 10.1 -> 6.9
// ms; a 64-slice slab of 2000^3 from 720 bf16 views 7.1 -> 5.0 ms; 64^3 30 -> 6 us.
//
// Everything else a view needs -- shift fraction, tap weights, crop offset --
// is one 16-byte entry of a per-CTA table in stream order (H = 2: 8 more bytes
// of weights), built once.  Views go block by block (D views): a block's end
// completes a decimated view and moves the running sums on.

constexpr int kCW = 16;       // shifted columns per warp
constexpr int kTP = kCW + 4;  // row pitch of the transpose buffer (floats; 5 16-byte units: no conflicts)
// Column segments (consumer warps) per CTA; wider squares take several CTAs.
// With the producer 8 warps, so that three CTAs (H = 1) or two (H = 2) share an
// SM's registers; nine warps leave room for two and one.  Squares of 113-128
// columns, 8 segments in one CTA against 4 + 4: 280^3 x 400 f32 156 -> 115 us,
// 300^3 x 420 2D taps 244 -> 177 us, 600^3 x 720 f32 1704 -> 1581 us.
constexpr int kDecMaxSegs = 7;
// Warps that the registers of an SM hold (80 and 128 a thread, see the kernel)
template <int H>
constexpr int kDecSmWarps = H == 1 ? 24 : 16;
static_assert((kDecMaxSegs + 1) * 3 <= kDecSmWarps<1> && (kDecMaxSegs + 1) * 2 <= kDecSmWarps<2>,
              "whole CTAs fill an SM's registers");
// ring shape per element type and tap length: slots of kG views, kStages slots.
// float32, measured at 512^3: what counts is that the CTAs the registers allow
// fit an SM (three with H = 1: 4 x 1 views are 16 % slower than 3 x 1; two with
// H = 2: 3 x 1 4 % slower than 4 x 1).  16-bit, 2000^3: fewer waits (3 x 2 views 4 %
// slower than 2 x 3, 2 x 2 6 %, 6 x 1 10 %).
template <typename TQ, int H>
struct Ring {
    static constexpr int kG = sizeof(TQ) == 4 ? 1 : 3, kStages = sizeof(TQ) == 4 ? (H == 1 ? 3 : 4) : 2;
};
// The last segment's 16-byte loads run past a row's end where the square uses
// few of its columns: up to 32 bytes (float32, one or five columns used, the crop
// three columns into its box: 20 columns read, 12 staged), in the last row of
// the last box past the ring.
constexpr int kRingSlack = 128;
constexpr uint64_t kDecWaitNs = 2000000000ull;

// Per-CTA tables over the stream of decimated views j0 .. j1 - 1: position
// pos is view k' = j0 D - (H D - 1) + pos (taken mod P), s_v[pos] = {shift
// fraction, the crop's offset inside its aligned box, weights 0 and 1}, s_w2[pos] = weights 2 and 3 (H = 2),
// s_c[pos] = crop column.
template <int kAl, int H>
__device__ __forceinline__ void build_stream_table(float4 *s_v, float2 *s_w2, int *s_c,
                                                   const int32_t *__restrict__ crop,
                                                   const GeomEntry *__restrict__ geo,
                                                   const float4 *__restrict__ tapw, int q, int P, int D, int j0,
                                                   int nstream) {
    for (int pos = threadIdx.x; pos < nstream; pos += blockDim.x) {
        const int kp = j0 * D + pos - (H * D - 1);
        const int kk = ((kp % P) + P) % P;
        const int c = crop[(size_t)q * P + kk];
        const int jb = floor_div(kp, D);
        const int r = kp - jb * D;
        const float4 w = tapw[r];
        s_v[pos] = make_float4(geo[(size_t)q * P + kk].frac, __int_as_float(c & (kAl - 1)), w.x, w.y);
        if (H == 2) s_w2[pos] = make_float2(w.z, w.w);
        s_c[pos] = c;
    }
}

// 16 bytes of a row, as floats
template <typename TQ>
struct Row16;
template <>
struct Row16<float> {
    static constexpr int kN = 4;
    static __device__ __forceinline__ void load(uint32_t a, float *v) {
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                     : "r"(a)
                     : "memory");
    }
};
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 u;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w)
                 : "r"(a)
                 : "memory");
    return u;
}
template <>
struct Row16<__nv_bfloat16> {
    static constexpr int kN = 8;
    static __device__ __forceinline__ void load(uint32_t a, float *v) {
        const uint4 u = lds128(a);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // bfloat16 is the top half of a float32
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};
template <>
struct Row16<__half> {
    static constexpr int kN = 8;
    static __device__ __forceinline__ void load(uint32_t a, float *v) {
        const uint4 u = lds128(a);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
            v[2 * i] = f.x;
            v[2 * i + 1] = f.y;
        }
    }
};

// One view for one lane: its row's samples at columns OFF .. OFF + kCW of the
// 16-byte aligned address a feed the 2H running sums of its kCW columns.
template <typename TQ, int H, int OFF>
__device__ __forceinline__ void view_step(uint32_t a, float f, const float (&w)[2 * H], float (&acc)[2 * H][kCW]) {
    constexpr int kN = Row16<TQ>::kN;
    constexpr int kL = (OFF + kCW + 1 + kN - 1) / kN;
    float v[kL * kN];
#pragma unroll
    for (int i = 0; i < kL; ++i) Row16<TQ>::load(a + 16u * (uint32_t)i, v + i * kN);
#pragma unroll
    for (int i = 0; i < kCW; ++i) {
        const float smp = fmaf(f, v[OFF + i + 1] - v[OFF + i], v[OFF + i]);
#pragma unroll
        for (int m = 0; m < 2 * H; ++m) acc[m][i] = fmaf(w[m], smp, acc[m][i]);
    }
}

template <typename TQ, int H>
__device__ __forceinline__ void view_any(int off, uint32_t a, float f, const float (&w)[2 * H],
                                         float (&acc)[2 * H][kCW]) {
    switch (off) {
        case 0: view_step<TQ, H, 0>(a, f, w, acc); break;
        case 1: view_step<TQ, H, 1>(a, f, w, acc); break;
        case 2: view_step<TQ, H, 2>(a, f, w, acc); break;
        case 3: view_step<TQ, H, 3>(a, f, w, acc); break;
        default:
            if constexpr (sizeof(TQ) == 2) {
                switch (off) {
                    case 4: view_step<TQ, H, 4>(a, f, w, acc); break;
                    case 5: view_step<TQ, H, 5>(a, f, w, acc); break;
                    case 6: view_step<TQ, H, 6>(a, f, w, acc); break;
                    default: view_step<TQ, H, 7>(a, f, w, acc); break;
                }
            }
    }
}

// dynamic shared memory: ring, transpose buffers, tables
__host__ __device__ inline size_t dec_smem(int es, int stages, int tile_stride, int warps, int nstream, int H) {
    return 128 + (size_t)es * stages * tile_stride + kRingSlack + (size_t)warps * 32 * kTP * sizeof(float) +
           (size_t)nstream * (16 + (H == 2 ? 8 : 0) + 4);
}

// the thread bound only sets the register limit: 80 (24 warps per SM) for the
// two running sums of the triangle, 128 (16 warps) for the four of 2D-tap filters
template <typename TQ, int H>
__global__ void __launch_bounds__(32 * kDecSmWarps<H>, 1)
decompose_rows_kernel(const __grid_constant__ CUtensorMap tmap, float *__restrict__ Sp,
                      const int32_t *__restrict__ crop, const GeomEntry *__restrict__ geo,
                      const int32_t *__restrict__ Tq, const float4 *__restrict__ tapw, int *status, int Tstride,
                      int P, int D, int Pd, int Nv, int Wc, int tile_stride, int segs, int chunks, int rowoff, int rowend,
                      int jrange) {
    constexpr int ES = (int)sizeof(TQ);
    constexpr int kAlign = 16 / ES;
    constexpr int kG = Ring<TQ, H>::kG, kStages = Ring<TQ, H>::kStages;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *ring = smem_raw + ((128u - (tma::smem_u32(smem_raw) & 127u)) & 127u);
    const uint32_t tile_bytes = (uint32_t)(ES * tile_stride);
    const int j0 = blockIdx.z * jrange, j1 = min(j0 + jrange, Pd);
    // views streamed: k' = j0 D - (H D - 1) .. (j1 - 1) D + H D - 1 (view k' mod P)
    const int nstream = (j1 - j0) * D + (2 * H - 1) * D - 1;
    const int nstage = (nstream + kG - 1) / kG;
    const int warps = (int)(blockDim.x >> 5) - 1;  // consumer warps
    float *tbuf = (float *)(ring + (size_t)tile_bytes * kStages * kG + kRingSlack);
    float4 *s_v = (float4 *)(tbuf + (size_t)warps * 32 * kTP);
    float2 *s_w2 = (float2 *)(s_v + nstream);
    int *s_c = (int *)(s_w2 + (H == 2 ? nstream : 0));
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages];

    const int q = blockIdx.x / chunks;
    const int tc = (blockIdx.x - q * chunks) * (segs * kCW);  // first column of the CTA's segments
    const int band = 32 * (warps / segs);                     // rows per CTA
    const int v0 = rowoff + blockIdx.y * band;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    build_stream_table<kAlign, H>(s_v, s_w2, s_c, crop, geo, tapw, q, P, D, j0, nstream);
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            tma::mbar_init(&full[i], 1);
            tma::mbar_init(&empty[i], warps);
        }
        tma::fence_mbar_init();
    }
    __syncthreads();

    if (warp == warps) {  // producer
        if (lane != 0) return;
        int kk = ((j0 * D - (H * D - 1)) % P + P) % P, n = 0, slot = 0;
        uint32_t phase = 0;  // parity of the slot's current round
        for (; n < nstage; ++n) {
            // round r of a slot may start once its round r - 1 was consumed
            if (n >= kStages && !tma::mbar_wait_bounded(&empty[slot], phase ^ 1u, kDecWaitNs)) {
                atomicOr(status, 2);
                break;
            }
            const int nv = min(kG, nstream - n * kG);
            tma::fence_proxy_async();
            tma::mbar_arrive_expect_tx(&full[slot], (uint32_t)(nv * band * Wc * ES));
            for (int w = 0; w < nv; ++w) {
                tma::load_3d(ring + (size_t)tile_bytes * (slot * kG + w), &tmap, &full[slot],
                             (s_c[n * kG + w] & ~(kAlign - 1)) + tc, v0, kk);
                if (++kk == P) kk = 0;
            }
            if (++slot == kStages) {
                slot = 0;
                phase ^= 1u;
            }
        }
        // copies still in flight must land before the CTA may exit
        for (int m = max(0, n - kStages); m < n; ++m)
            tma::mbar_wait_bounded(&full[m % kStages], (uint32_t)((m / kStages) & 1), kDecWaitNs);
        return;
    }

    const int grp = warp / segs, seg = warp - grp * segs;
    const int rib = 32 * grp;  // first of the warp's rows in the band
    const int t0 = tc + seg * kCW;  // first of its columns
    const int ncol = Tq[q] - t0;  // columns of the warp that the square has
    float acc[2 * H][kCW];
#pragma unroll
    for (int m = 0; m < 2 * H; ++m)
#pragma unroll
        for (int i = 0; i < kCW; ++i) acc[m][i] = 0.f;
    // coalesced store: lane writes 16 bytes at row rib + lane / 4 (+ 8, 16, 24), column t0 + 4 (lane % 4)
    const size_t vstride = (size_t)Nv * Tstride;
    const int srow = v0 + rib + (lane >> 2), scol = t0 + 4 * (lane & 3);
    float *o = Sp + ((size_t)((size_t)q * Pd + j0) * Nv + srow) * Tstride + scol;
    float *tb = tbuf + (size_t)warp * 32 * kTP;
    const uint32_t lane_addr = tma::smem_u32(ring) + (uint32_t)(ES * ((rib + lane) * Wc + seg * kCW));
    int slot = 0;
    uint32_t phase = 0;

    // the stream starts at the second view of block j0 - H, whose end completes view j0 - 2 H + 1
    int left = D - 1, w = 0;
    const float4 *pe = s_v;
    const float2 *pe2 = s_w2;
    uint32_t a = lane_addr;
    for (int jst = j0 - 2 * H + 1; jst < j1; ++jst, left = D) {
#pragma unroll 1
        for (; left > 0; --left) {
            const float4 e = *pe++;
            float wt[2 * H];
            wt[0] = e.z;
            wt[1] = e.w;
            if constexpr (H == 2) {
                const float2 e2 = *pe2++;
                wt[2] = e2.x;
                wt[3] = e2.y;
            }
            if (w == 0) {
                const bool ok = tma::mbar_wait_bounded(&full[slot], phase, kDecWaitNs);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) atomicOr(status, 2);
                    return;
                }
            }
            view_any<TQ, H>(__float_as_int(e.y), a, e.x, wt, acc);
            a += tile_bytes;
            if (++w == kG) {
                w = 0;
                __syncwarp();
                if (lane == 0) tma::mbar_arrive(&empty[slot]);
                if (++slot == kStages) {
                    slot = 0;
                    phase ^= 1u;
                    a = lane_addr;
                }
            }
        }
        if (jst >= j0) {  // decimated view jst is complete
            // zero past the square's T columns
#pragma unroll
            for (int i = 0; i < kCW; ++i)
                if (i >= ncol) acc[0][i] = 0.f;
            float4 *dst = (float4 *)(tb + lane * kTP);
#pragma unroll
            for (int i = 0; i < kCW; i += 4)
                dst[i / 4] = make_float4(acc[0][i], acc[0][i + 1], acc[0][i + 2], acc[0][i + 3]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 val = *(const float4 *)(tb + (8 * i + (lane >> 2)) * kTP + 4 * (lane & 3));
                if (srow + 8 * i < rowend && scol < Tstride) *(float4 *)(o + (size_t)(8 * i) * Tstride) = val;
            }
            o += vstride;
            __syncwarp();
        }
#pragma unroll
        for (int i = 0; i < kCW; ++i) {
#pragma unroll
            for (int m = 0; m < 2 * H - 1; ++m) acc[m][i] = acc[m + 1][i];
            acc[2 * H - 1][i] = 0.f;
        }
    }
}

// Share of its rate that an SM reaches with w resident consumer warps (512^3
// f32: 7, 14 and 21 of them)
double sm_rate(double w) {
    return w <= 7.0    ? 0.59 * w / 7.0
           : w <= 14.0 ? 0.59 + 0.27 * (w - 7.0) / 7.0
                       : std::min(1.0, 0.86 + 0.14 * (w - 14.0) / 7.0);
}

// Rows of a launch: the arrays hold `layout` rows per view (S' included)
// and the launch covers rows rowoff .. rowend - 1 of them.
struct Rows {
    int layout, rowoff, rowend;
};

// Shape of the staged kernel's launch over `nrows` detector rows.
struct RowsShape {
    int Wc, tile_stride;              // columns of a crop box; elements per staged box
    int segs, chunks, warps;          // column segments per CTA, CTAs side by side, consumer warps
    int band, bands;                  // rows per CTA, bands of rows
    int jrange, resident;             // decimated views per CTA; CTAs that an SM holds at once
    size_t smem;
};

// False where the staged kernel does not apply: Q's rows must be whole 16-byte
// units, D <= 128 and the ring plus the stream tables fit in shared memory.
template <typename TQ, int H>
bool rows_shape(const PlanImpl &p, int nrows, RowsShape &r) {
    constexpr int kAlign = 16 / (int)sizeof(TQ);
    if ((p.g.Nu % kAlign) != 0 || p.D > kMaxTapD) return false;
    const int all = (p.Tstride + kCW - 1) / kCW;  // column segments of a square
    // as few CTAs side by side as hold them, or one more where that leaves fewer
    // segments empty: 16 segments 4 x 4 rather than 3 x 6 (584^3 x 720, s = 2: 865 ->
    // 795 us, 2D taps 1243 -> 992), 9 as 3 x 3 rather than 2 x 5 (660^3 x 400 1107 ->
    // 1030 us, 2D taps 1766 -> 1392), but 13 as 2 x 7 (256^3 x 360, s = 1: 56 us, 57 in 3 x 5)
    r.chunks = (all + kDecMaxSegs - 1) / kDecMaxSegs;
    auto segs_of = [&](int chunks) { return (all + chunks - 1) / chunks; };
    if ((r.chunks + 1) * segs_of(r.chunks + 1) < r.chunks * segs_of(r.chunks)) ++r.chunks;
    r.segs = segs_of(r.chunks);
    // the segments' columns + neighbour + crop offset, whole 16-byte units, an odd number of them
    r.Wc = (std::min(p.od.Tmax, r.segs * kCW) + 1 + (kAlign - 1) + (kAlign - 1)) & ~(kAlign - 1);
    if ((r.Wc / kAlign) % 2 == 0) r.Wc += kAlign;
    // narrow squares: several row groups per CTA, at least four consumer warps
    const int groups = std::max(1, std::min((nrows + 31) / 32, 4 / r.segs));
    r.warps = r.segs * groups;
    r.band = 32 * groups;
    r.bands = (nrows + r.band - 1) / r.band;
    r.tile_stride = (r.band * r.Wc + 63) & ~63;  // elements; 128-byte multiple for every type
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr int kLead = 2 * H - 1;  // a range streams kLead D - 1 views besides its own
    auto smem_of = [&](int jr) {
        return dec_smem((int)sizeof(TQ), Ring<TQ, H>::kStages * Ring<TQ, H>::kG, r.tile_stride, r.warps,
                        (jr + kLead) * p.D - 1, H);
    };
    // The decimated views are split into ranges (the same sums in the same
    // order, so the same result), by a model of the time of the SM with the
    // most CTAs: as many of them at once as its registers and shared memory
    // hold (a shorter table can let one more fit), wave after wave, each wave
    // the views its CTAs stream at the rate of its resident warps; and a fifth
    // of a CTA more, for CTAs that don't end together.  Of 148 shapes (37 sizes
    // from 64^3 to 1000^3, float32 and bfloat16, both tap lengths) measured with
    // 1 to 64 ranges of at least 4 kLead views, the choice is 0.4 % behind the
    // best one in the mean.  Small grids take ranges down to one view (of 4
    // kLead or more: 128^3 x 128 bf16, D = 8, 2D taps 58 us against 19).
    const long long ctas = (long long)p.od.nsq * r.chunks * r.bands;
    int per_sm = 0;
    if (cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) return false;
    r.resident = 0;
    double best = 0.0;
    for (int n = 1; n <= std::min(64, p.Pd); ++n) {
        const int jr = (p.Pd + n - 1) / n;
        const size_t smem = smem_of(jr);
        const int fit = std::min(kDecSmWarps<H> / (r.warps + 1), (int)((size_t)per_sm / (smem + 2048)));
        if (fit < 1 || smem > 200 * 1024) continue;
        const long long per = (ctas * ((p.Pd + jr - 1) / jr) + sms - 1) / sms;  // CTAs of an SM, at most
        const long long rest = per % fit;
        const double last = rest ? (double)rest / sm_rate((double)rest * r.warps) : 0.0;
        const double waves = (double)(per - rest) / sm_rate((double)fit * r.warps) + last;
        const double cost = (waves + 0.2) * ((jr + kLead) * p.D + 1);
        if (r.resident == 0 || cost < best) {
            best = cost;
            r.jrange = jr;
            r.resident = fit;
            r.smem = smem;
        }
    }
    return r.resident > 0 && r.bands <= 65535;
}

// The staged kernel, where it applies and Q and S' are 16-byte aligned (bulk
// copies, vector stores).
template <typename TQ, int H>
cudaError_t try_rows(const PlanImpl &p, const TQ *Q, float *out, cudaStream_t st, Rows rw, bool &launched) {
    launched = false;
    RowsShape r;
    if (((uintptr_t)Q & 15) != 0 || ((uintptr_t)out & 15) != 0) return cudaSuccess;
    if (!rows_shape<TQ, H>(p, rw.rowend - rw.rowoff, r)) return cudaSuccess;
    CUtensorMap map;
    const uint64_t dims[3] = {(uint64_t)p.g.Nu, (uint64_t)rw.layout, (uint64_t)p.g.P};
    const uint64_t strides[2] = {(uint64_t)p.g.Nu * sizeof(TQ), (uint64_t)p.g.Nu * rw.layout * sizeof(TQ)};
    const uint32_t box[3] = {(uint32_t)r.Wc, (uint32_t)r.band, 1u};
    const CUtensorMapDataType dt = sizeof(TQ) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : (std::is_same<TQ, __half>::value ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                                      : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
    if (encode_map_3d(&map, dt, Q, dims, strides, box) != cudaSuccess) return cudaSuccess;
    launched = true;
    cudaError_t e = ensure_smem<decompose_rows_kernel<TQ, H>>(r.smem);
    if (e != cudaSuccess) return e;
    dim3 grid(p.od.nsq * r.chunks, r.bands, (p.Pd + r.jrange - 1) / r.jrange);
    decompose_rows_kernel<TQ, H><<<grid, 32 * (r.warps + 1), r.smem, st>>>(
        map, out, p.od.crop, p.od.geo, p.od.T, p.tapw, p.status, p.Tstride, p.g.P, p.D, p.Pd, rw.layout, r.Wc,
        r.tile_stride, r.segs, r.chunks, rw.rowoff, rw.rowend, r.jrange);
    return cudaGetLastError();
}

constexpr int kBandRows = kGenWarps * kGenRows;  // rows per CTA of the generic kernel

// Decimated views per CTA of the generic kernel, from the `ctas` of one range:
// up to eight CTAs per SM, by the views that a CTA streams times the CTAs of an
// SM, of which `idle` run as fast as one: eight, or three where 2D taps (four
// running sums) meet a small grid.  49^3 x 72 bf16, D = 6, 2D taps: 27 us where a
// range had to have twice the blocks that it streams besides its own, 15 now;
// 331^3 x 328 f32 333 us, both.
int generic_range(const PlanImpl &p, long long ctas) {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int most = (int)std::min<long long>(p.Pd, (8LL * sms + ctas - 1) / ctas);
    const double idle = p.tap_blocks == 2 && ctas < 2LL * sms ? 3.0 : 8.0;
    int jrange = p.Pd;
    double best = 0.0;
    for (int n = 1; n <= most; ++n) {
        const int jr = (p.Pd + n - 1) / n;
        const double per = (double)(ctas * ((p.Pd + jr - 1) / jr)) / sms;
        const double cost = (jr + 2 * p.tap_blocks - 1) * std::max(idle, per);
        if (n == 1 || cost < best) {
            best = cost;
            jrange = jr;
        }
    }
    return jrange;
}

template <typename TQ, int H>
cudaError_t form_t(const PlanImpl &p, fdkod_forms &f) {
    RowsShape r;
    if (!rows_shape<TQ, H>(p, p.g.Nv, r)) {
        const int tiles = (p.Tstride + 31) / 32, bands = (p.g.Nv + kBandRows - 1) / kBandRows;
        const int jrange = generic_range(p, (long long)tiles * bands * p.od.nsq);
        f.dec_ranges = (p.Pd + jrange - 1) / jrange;
        return cudaSuccess;
    }
    f.dec_warps = r.warps;
    f.dec_ranges = (p.Pd + r.jrange - 1) / r.jrange;
    f.dec_resident = r.resident;
    cudaError_t e = ensure_smem<decompose_rows_kernel<TQ, H>>(r.smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f.dec_occupancy, decompose_rows_kernel<TQ, H>,
                                                         32 * (r.warps + 1), r.smem);
}

template <typename TQ>
cudaError_t launch_t(const PlanImpl &p, const TQ *Q, float *out, cudaStream_t st, Rows rw) {
    if (p.tap_blocks != 1 && p.tap_blocks != 2) return cudaErrorInvalidValue;
    bool launched = false;
    cudaError_t te = p.tap_blocks == 2 ? try_rows<TQ, 2>(p, Q, out, st, rw, launched)
                                       : try_rows<TQ, 1>(p, Q, out, st, rw, launched);
    if (launched || te != cudaSuccess) return te;
    const int tiles = (p.Tstride + 31) / 32, bands = (rw.rowend - rw.rowoff + kBandRows - 1) / kBandRows;
    const int jrange = generic_range(p, (long long)tiles * bands * p.od.nsq);
    const dim3 grid(tiles * ((p.Pd + jrange - 1) / jrange), bands, p.od.nsq);
    const dim3 block(32, kGenWarps);
    auto kernel = p.tap_blocks == 2 ? decompose_kernel<TQ, 2> : decompose_kernel<TQ, 1>;
    kernel<<<grid, block, 0, st>>>(Q, out, p.od.crop, p.od.geo, p.od.T, p.tapw, p.Tstride, p.g.P, p.D, p.Pd, rw.layout,
                                   p.g.Nu, rw.rowoff, rw.rowend, tiles, jrange);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_decompose(const PlanImpl &p, const void *Q, float *out, cudaStream_t st, Band b) {
    const int nrows = b.nrows < 0 ? p.g.Nv : b.nrows;
    Rows rw{nrows, 0, nrows};
    if (b.whole_arrays) rw = Rows{p.g.Nv, b.row0, b.row0 + nrows};
    if (p.net) {
        if (b.whole_arrays && (b.row0 != 0 || nrows != p.g.Nv)) return cudaErrorInvalidValue;
        return launch_net_decompose(p, Q, out, st, nrows);
    }
    switch (p.qtype) {
        case FDKOD_F32: return launch_t(p, (const float *)Q, out, st, rw);
        case FDKOD_BF16: return launch_t(p, (const __nv_bfloat16 *)Q, out, st, rw);
        case FDKOD_F16: return launch_t(p, (const __half *)Q, out, st, rw);
    }
    return cudaErrorInvalidValue;
}

cudaError_t decompose_form(const PlanImpl &p, fdkod_forms &f) {
    if (p.D == 1 || p.net) return cudaSuccess;
    const bool wide = p.tap_blocks == 2;
    switch (p.qtype) {
        case FDKOD_F32: return wide ? form_t<float, 2>(p, f) : form_t<float, 1>(p, f);
        case FDKOD_BF16: return wide ? form_t<__nv_bfloat16, 2>(p, f) : form_t<__nv_bfloat16, 1>(p, f);
        case FDKOD_F16: return wide ? form_t<__half, 2>(p, f) : form_t<__half, 1>(p, f);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fdkod
