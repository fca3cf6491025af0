// HBM-bound kernels of the layer: LayerNorm forward, LayerNorm backward (fused with the
// residual-gradient add and two bias-gradient column sums), column sums, and the row-dot
// preprocess of the attention backward.  All use 16-byte accesses (8 bf16 per thread per
// access), fp32 arithmetic, warp shuffles plus one shared-memory hop for row reductions, and
// fixed-order two-stage reductions for anything summed over tokens (bitwise reproducible).
#include <algorithm>
#include <map>
#include <mutex>

#include "pw_kernels.h"

namespace pw {
namespace {

constexpr int kMaxWarps = 8;          // CTAs have at most 256 threads
constexpr int kRowThreadsMax = 256;

// A row of d elements is handled by tpr = d / (8*CHUNKS) threads, CHUNKS 16-byte pieces each;
// thread i of the row owns columns 8*(i + j*tpr) .. +7 for j < CHUNKS (coalesced per j).
struct RowPlan { int chunks, tpr, rows_per_cta, threads; };
bool plan_rows(int d, RowPlan* rp)
{
    for (int c = 1; c <= 4; c *= 2) {
        if (d % (8 * c * 32) != 0) continue;
        int tpr = d / (8 * c);
        if (tpr > kRowThreadsMax) continue;
        rp->chunks = c; rp->tpr = tpr;
        rp->rows_per_cta = kRowThreadsMax / tpr;
        rp->threads = rp->rows_per_cta * tpr;
        return true;
    }
    return false;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void unpack8_pairs(const uint4& v, uint64_t* p)
{
    p[0] = pack_f32x2(bf16_lo(v.x), bf16_hi(v.x)); p[1] = pack_f32x2(bf16_lo(v.y), bf16_hi(v.y));
    p[2] = pack_f32x2(bf16_lo(v.z), bf16_hi(v.z)); p[3] = pack_f32x2(bf16_lo(v.w), bf16_hi(v.w));
}
__device__ __forceinline__ uint32_t pack_pair_bf16(uint64_t p)
{
    float lo, hi;
    unpack_f32x2(p, lo, hi);
    return pack_bf16(lo, hi);
}
__device__ __forceinline__ uint64_t splat2(float v) { return pack_f32x2(v, v); }

// LayerNorm forward.  A row is handled by W warps (W = 1 for d <= 2048), each lane holding CH
// 16-byte pieces (lane i of warp w owns columns 8*(i + 32*(w + W*j)) .. +7, j < CH): all of a
// lane's loads are issued at once, the statistics need only warp shuffles (plus one shared-memory
// hop when W > 1).  256-thread CTAs hold 8/W rows.
// FEW: no more CTAs than SMs.  gamma and beta then travel with the row, for a second trip behind the sums is a good part of the time;
// with more CTAs the registers that takes cost more.  us, later -> with the row: 1024 x 512 1.97 -> 1.68, 1024 x 1024 2.59 -> 2.09; with 80 registers for
// all 2048 x 1024 2.80 -> 3.17, 8192 x 1024 7.8 -> 8.4.
template <int CH, bool FEW>
__global__ void __launch_bounds__(kRowThreadsMax, FEW ? 1 : 3)
ln_fwd_kernel(const __nv_bfloat16* x, const __nv_bfloat16* gamma,
              const __nv_bfloat16* beta, int T, int d, float eps, __nv_bfloat16* h,
              float* mu, float* rstd, int W)
{
    __shared__ float red[2][kMaxWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows_per_cta = kMaxWarps / W;
    const int row_in_cta = warp / W, wr = warp % W;
    const int row = blockIdx.x * rows_per_cta + row_in_cta;
    const bool live = row < T && row_in_cta < rows_per_cta;
    grid_dep_wait();
    grid_dep_launch();                                  // in this order: see kOrderWeightsReady
    // two-wide fp32 throughout: neighbouring columns share a 64-bit register
    uint64_t v[CH][4];
    uint64_t acc = 0ull;
    uint4 raw[CH], gb[FEW ? CH : 1][2];
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        const int col = 8 * (lane + 32 * (wr + W * j));
        raw[j] = live ? *reinterpret_cast<const uint4*>(x + static_cast<size_t>(row) * d + col) : make_uint4(0, 0, 0, 0);
    }
    if constexpr (FEW) {
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            const int col = 8 * (lane + 32 * (wr + W * j));
            gb[j][0] = *reinterpret_cast<const uint4*>(gamma + col);
            gb[j][1] = *reinterpret_cast<const uint4*>(beta + col);
        }
    }
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        unpack8_pairs(raw[j], v[j]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc = fadd2(acc, v[j][k]);
    }
    float a0, a1;
    unpack_f32x2(acc, a0, a1);
    float s = warp_sum(a0 + a1);
    if (W > 1) {
        if (lane == 0) red[0][warp] = s;
        __syncthreads();
        s = 0.f;
        for (int i = 0; i < W; ++i) s += red[0][row_in_cta * W + i];
    }
    const float mean = s / d;
    const uint64_t nmean = splat2(-mean);
    acc = 0ull;
#pragma unroll
    for (int j = 0; j < CH; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) { const uint64_t c = fadd2(v[j][k], nmean); acc = ffma2(c, c, acc); }
    unpack_f32x2(acc, a0, a1);
    float q = warp_sum(a0 + a1);
    if (W > 1) {
        if (lane == 0) red[1][warp] = q;
        __syncthreads();
        q = 0.f;
        for (int i = 0; i < W; ++i) q += red[1][row_in_cta * W + i];
    }
    const float r = rsqrtf(q / d + eps);
    if (!live) return;
    const uint64_t r2 = splat2(r), nmr2 = splat2(-mean * r);
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        const int col = 8 * (lane + 32 * (wr + W * j));
        uint64_t g[4], b[4];
        unpack8_pairs(FEW ? gb[FEW ? j : 0][0] : *(reinterpret_cast<const uint4*>(gamma + col)), g);
        unpack8_pairs(FEW ? gb[FEW ? j : 0][1] : *(reinterpret_cast<const uint4*>(beta + col)), b);
        uint4 o;
        o.x = pack_pair_bf16(ffma2(ffma2(v[j][0], r2, nmr2), g[0], b[0]));
        o.y = pack_pair_bf16(ffma2(ffma2(v[j][1], r2, nmr2), g[1], b[1]));
        o.z = pack_pair_bf16(ffma2(ffma2(v[j][2], r2, nmr2), g[2], b[2]));
        o.w = pack_pair_bf16(ffma2(ffma2(v[j][3], r2, nmr2), g[3], b[3]));
        *reinterpret_cast<uint4*>(h + static_cast<size_t>(row) * d + col) = o;
    }
    if (wr == 0 && lane == 0) { mu[row] = mean; rstd[row] = r; }
}

__global__ void __launch_bounds__(256)
affine_f32_kernel(const float* x, long long n, float scale, float shift, float* y)
{
    grid_dep_launch();
    grid_dep_wait();
    const long long i = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
    if (i < n) y[i] = fmaf(x[i], scale, shift);
}

// a = GeLU(u) on bf16 tensors: the backward pass of a layer that did not keep `a` re-derives it from
// the pre-activations it did keep.  8 elements per thread and iteration; 4 bytes per element.
__device__ __forceinline__ uint4 gelu8(const uint4& w, int act)
{
    const uint32_t in[4] = {w.x, w.y, w.z, w.w};
    uint32_t out[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float lo = __uint_as_float(in[q] << 16), hi = __uint_as_float(in[q] & 0xffff0000u);
        gelu2(lo, hi, act);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(out[q]) : "f"(hi), "f"(lo));
    }
    return make_uint4(out[0], out[1], out[2], out[3]);
}

__global__ void __launch_bounds__(256)
gelu_fwd_kernel(const __nv_bfloat16* u, __nv_bfloat16* a, long long n8, int act)
{
    grid_dep_launch();
    grid_dep_wait();
    const long long stride = static_cast<long long>(gridDim.x) * 256;
    long long i = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
    for (; i + 3 * stride < n8; i += 4 * stride) {                    // four loads in flight per thread
        uint4 w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = __ldcs(reinterpret_cast<const uint4*>(u + (i + j * stride) * 8));
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(a + (i + j * stride) * 8) = gelu8(w[j], act);
    }
    for (; i < n8; i += stride)
        *reinterpret_cast<uint4*>(a + i * 8) = gelu8(*reinterpret_cast<const uint4*>(u + i * 8), act);
}

// W warps per row and CH pieces per lane for a row of d elements (d a multiple of 256).
bool plan_warp_rows(int d, int* W, int* CH)
{
    if (d % 256 != 0) return false;
    const int total = d / 256;
    for (int w = 1; w <= kMaxWarps; ++w)
        if (total % w == 0 && total / w <= 8 && kMaxWarps % w == 0) { *W = w; *CH = total / w; return true; }
    return false;
}

// LayerNorm backward.  Persistent over rows; every thread keeps the column sums of its own
// columns in registers; they leave at the end as one partial row per CTA:
// partials[cta][4][d] = {dgamma, dbeta, sum resid, sum dx} (its row slots' sums added in slot order).
// The next row's three inputs are fetched before the current row's reduction, and the two row
// sums share one barrier.
// rows in the prefetch ring (six were measured slower than four at every width)
__host__ __device__ constexpr int ln_bwd_depth(int) { return 4; }
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src, bool valid)
{
    const int n = valid ? 16 : 0;                       // 0: the 16 bytes are zero-filled, src is not read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The kernel is bound by instruction issue as much as by memory, so all element-wise arithmetic
// is two-wide fp32 (values of neighbouring columns packed in one 64-bit register).
// BIAS_SUMS: also produce the column sums of the residual gradient and of dx (the two bias
// gradients that the LN2 backward of a layer yields for free); without them the partial rows hold
// two quantities instead of four.
template <int CHUNKS, bool BIAS_SUMS>
__global__ void __launch_bounds__(kRowThreadsMax, CHUNKS == 1 ? 2 : 1)
ln_bwd_kernel(const __nv_bfloat16* dh, const __nv_bfloat16* x,
              const float* mu, const float* rstd, const __nv_bfloat16* gamma,
              const __nv_bfloat16* resid, int T, int d, __nv_bfloat16* dx,
              float* partials, int tpr, int rows_per_cta)
{
    constexpr int kDepth = ln_bwd_depth(CHUNKS);
    __shared__ float red[2][2][kMaxWarps];
    const int row_in_cta = threadIdx.x / tpr, tr = threadIdx.x % tpr;
    const int wpr = tpr >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    grid_dep_wait();
    grid_dep_launch();                                  // in this order: kernels that start late may follow (see launch_wgrad)
    uint64_t gm[CHUNKS][4];
    uint64_t acc_g[CHUNKS][4], acc_b[CHUNKS][4], acc_r[CHUNKS][4], acc_x[CHUNKS][4];
#pragma unroll
    for (int j = 0; j < CHUNKS; ++j) {
        unpack8_pairs(*(reinterpret_cast<const uint4*>(gamma + 8 * (tr + j * tpr))), gm[j]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc_g[j][k] = acc_b[j][k] = acc_r[j][k] = acc_x[j][k] = 0ull;
    }
    const int row_groups = (T + rows_per_cta - 1) / rows_per_cta;
    // The three inputs of the rows this thread will handle travel through a private ring in
    // shared memory, kDepth - 1 rows ahead (16-byte asynchronous copies; a thread only ever
    // reads what it fetched itself, so no barrier is involved).  Slot (stage, input, j) of thread
    // t is ring[((stage * 3 + input) * CHUNKS + j) * blockDim.x + t].
    extern __shared__ uint4 ln_bwd_ring[];
    const uint32_t ring0 = smem_u32(ln_bwd_ring) + 16u * threadIdx.x;
    const uint32_t slot_stride = 16u * blockDim.x;
    // Rows are visited with a constant stride, so the element offsets of the row being fetched and of
    // the row being computed are running sums (no 64-bit multiply per row).
    const int row_step = gridDim.x * rows_per_cta;
    const size_t off_step = static_cast<size_t>(row_step) * d;
    int pf_row = blockIdx.x * rows_per_cta + row_in_cta;                 // next row to fetch
    size_t pf_off = static_cast<size_t>(pf_row) * d + 8 * tr;
    auto issue = [&](int stage) {
        const bool live = pf_row < T;
#pragma unroll
        for (int j = 0; j < CHUNKS; ++j) {
            const size_t off = live ? pf_off + 8 * j * tpr : 0;
            const uint32_t dst = ring0 + (stage * 3 * CHUNKS + j) * slot_stride;
            cp_async_16(dst, dh + off, live);
            cp_async_16(dst + CHUNKS * slot_stride, x + off, live);
            cp_async_16(dst + 2 * CHUNKS * slot_stride, resid ? resid + off : dh + off, live && resid != nullptr);   // no residual: zeros
        }
        cp_async_commit();
        pf_row += row_step;
        pf_off += off_step;
    };
    float n_m = 0.f, n_r = 0.f;
    auto fetch_stats = [&](int rg) {
        const int row = rg * rows_per_cta + row_in_cta;
        const bool live = rg < row_groups && row < T;
        n_m = live ? mu[row] : 0.f;
        n_r = live ? rstd[row] : 0.f;
    };
#pragma unroll
    for (int s = 0; s < kDepth - 1; ++s) issue(s);
    fetch_stats(blockIdx.x);
    const float inv_d = 1.0f / d;
    int par = 0, stage = 0;
    int row = blockIdx.x * rows_per_cta + row_in_cta;
    size_t row_off = static_cast<size_t>(row) * d + 8 * tr;
    for (int rg = blockIdx.x; rg < row_groups; rg += gridDim.x, par ^= 1, row += row_step, row_off += off_step) {
        const bool live = row < T;
        const float r = n_r;
        const uint64_t r2 = splat2(r), nmr2 = splat2(-n_m * r);
        issue(stage == 0 ? kDepth - 1 : stage - 1);
        cp_async_wait<kDepth - 1>();                  // this row's copies have landed
        uint64_t xh[CHUNKS][4], g[CHUNKS][4], dhv[CHUNKS][4], rs[CHUNKS][4];
        uint64_t s1p = 0ull, s2p = 0ull;
#pragma unroll
        for (int j = 0; j < CHUNKS; ++j) {
            const uint4* slot = ln_bwd_ring + (stage * 3 * CHUNKS + j) * blockDim.x + threadIdx.x;
            unpack8_pairs(slot[0], dhv[j]);
            unpack8_pairs(slot[CHUNKS * blockDim.x], xh[j]);
            unpack8_pairs(slot[2 * CHUNKS * blockDim.x], rs[j]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                xh[j][k] = ffma2(xh[j][k], r2, nmr2);           // (x - mu) * rstd
                g[j][k] = fmul2(dhv[j][k], gm[j][k]);
                s1p = fadd2(s1p, g[j][k]);
                s2p = ffma2(g[j][k], xh[j][k], s2p);
            }
        }
        stage = stage + 1 == kDepth ? 0 : stage + 1;
        fetch_stats(rg + gridDim.x);
        float s1, s1b, s2, s2b;
        unpack_f32x2(s1p, s1, s1b);
        unpack_f32x2(s2p, s2, s2b);
        // Both sums in one set of exchanges: the lower half of the warp goes on with s1, the upper one with s2
        // (against two sets, with the reduce launch, us: 8192 x 2048 33.7 -> 33.1, 8192 x 1280 29.4 -> 28.4, 8192 x 8192 167 -> 162).
        const bool upper = lane >= 16;
        s1 += s1b; s2 += s2b;
        float v = upper ? s2 : s1;
        v += __shfl_xor_sync(0xffffffffu, upper ? s1 : s2, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (wpr > 1) {
            if ((lane & 15) == 0) red[par][lane >> 4][warp] = v;
            __syncthreads();
            // every lane takes one warp's partial sum; three exchange steps add up to eight of them
            const int src = lane & (kMaxWarps - 1);      // both groups of eight lanes of a half hold the same eight values
            v = src < wpr ? red[par][lane >> 4][row_in_cta * wpr + src] : 0.f;
#pragma unroll
            for (int o = kMaxWarps / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        }
        s1 = __shfl_sync(0xffffffffu, v, 0);
        s2 = __shfl_sync(0xffffffffu, v, 16);
        const uint64_t nmg2 = splat2(-s1 * inv_d), nmgx2 = splat2(-s2 * inv_d);
        if (live) {
#pragma unroll
            for (int j = 0; j < CHUNKS; ++j) {
                const size_t off = row_off + 8 * j * tpr;
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // dx = resid + rstd * (g - mean(g) - xh * mean(g * xh))
                    const uint64_t t = ffma2(xh[j][k], nmgx2, fadd2(g[j][k], nmg2));
                    w[k] = pack_pair_bf16(ffma2(r2, t, rs[j][k]));
                    // the bias gradient sums the values that are actually stored
                    if (BIAS_SUMS) acc_x[j][k] = fadd2(acc_x[j][k], pack_f32x2(bf16_lo(w[k]), bf16_hi(w[k])));
                    acc_g[j][k] = ffma2(dhv[j][k], xh[j][k], acc_g[j][k]);
                    acc_b[j][k] = fadd2(acc_b[j][k], dhv[j][k]);
                    if (BIAS_SUMS) acc_r[j][k] = fadd2(acc_r[j][k], rs[j][k]);
                }
                *reinterpret_cast<uint4*>(dx + off) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
    constexpr int NQ = BIAS_SUMS ? 4 : 2;
    float* prow = partials + static_cast<size_t>(blockIdx.x) * NQ * d;
    // Narrow rows (one piece per thread): the CTA's row slots add up first.  (Wider instances have one slot; with this code in them all the
    // same, 4096 tokens x 8192 took 95.1 us instead of 91.5.)
    if (CHUNKS == 1 && rows_per_cta > 1) {
        float* sums = reinterpret_cast<float*>(ln_bwd_ring);             // [slot][NQ][d], at most 8 K floats; the ring is idle
        cp_async_wait<0>();
        __syncthreads();
        float* mine = sums + (row_in_cta * NQ) * d + 8 * tr;
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            *reinterpret_cast<ulonglong2*>(mine + 2 * k) = make_ulonglong2(acc_g[0][k], acc_g[0][k + 1]);
            *reinterpret_cast<ulonglong2*>(mine + d + 2 * k) = make_ulonglong2(acc_b[0][k], acc_b[0][k + 1]);
            if (BIAS_SUMS) {
                *reinterpret_cast<ulonglong2*>(mine + 2 * d + 2 * k) = make_ulonglong2(acc_r[0][k], acc_r[0][k + 1]);
                *reinterpret_cast<ulonglong2*>(mine + 3 * d + 2 * k) = make_ulonglong2(acc_x[0][k], acc_x[0][k + 1]);
            }
        }
        __syncthreads();
        for (int c = 4 * threadIdx.x; c < NQ * d; c += 4 * blockDim.x) {
            float4 s = *reinterpret_cast<const float4*>(sums + c);
            for (int r = 1; r < rows_per_cta; ++r) {
                const float4 v = *reinterpret_cast<const float4*>(sums + r * NQ * d + c);
                s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
            }
            *reinterpret_cast<float4*>(prow + c) = s;
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < CHUNKS; ++j) {
        const int col = 8 * (tr + j * tpr);
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            // two pairs = four consecutive columns
            *reinterpret_cast<ulonglong2*>(prow + 0 * d + col + 2 * k) = make_ulonglong2(acc_g[j][k], acc_g[j][k + 1]);
            *reinterpret_cast<ulonglong2*>(prow + 1 * d + col + 2 * k) = make_ulonglong2(acc_b[j][k], acc_b[j][k + 1]);
            if (BIAS_SUMS) {
                *reinterpret_cast<ulonglong2*>(prow + 2 * d + col + 2 * k) = make_ulonglong2(acc_r[j][k], acc_r[j][k + 1]);
                *reinterpret_cast<ulonglong2*>(prow + 3 * d + col + 2 * k) = make_ulonglong2(acc_x[j][k], acc_x[j][k + 1]);
            }
        }
    }
}

// The same for few tokens: a CTA takes eight rows, a warp each, and is done.  A warp stages its row's three inputs at once
// (cp.async, no barrier: lanes read what they fetched), takes the row sums by shuffles and leaves dx in shared memory too; after the
// CTA's one barrier a thread owns columns and adds up the eight rows.  What bounds it is one trip to memory and the two
// hand-overs, where the persistent kernel above makes a trip, a barrier and two exchanges for every row of a slot.  Figures: ln_bwd_by_rows.
constexpr int kLnRows = 8;
constexpr int ln_rows_smem_bytes(int ch, bool sums) { return (sums ? 4 : 3) * kLnRows * 512 * ch; }      // dx stays there for its sums only
template <int CH, bool BIAS_SUMS>
__global__ void __launch_bounds__(32 * kLnRows)
ln_bwd_rows_kernel(const __nv_bfloat16* dh, const __nv_bfloat16* x, const float* mu, const float* rstd, const __nv_bfloat16* gamma,
                   const __nv_bfloat16* resid, int T, __nv_bfloat16* dx, float* partials)
{
    constexpr int d = 256 * CH, kPieces = d / 8;            // 16-byte pieces of a row
    extern __shared__ uint4 ln_rows_smem[];                 // [dh, x, resid, with BIAS_SUMS dx][row][piece]
    __shared__ float stats[kLnRows][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * kLnRows + warp;
    const bool live = row < T;
    uint4* mine = ln_rows_smem + warp * kPieces + lane;
    constexpr int kTensor = kLnRows * kPieces;
    grid_dep_wait();
    grid_dep_launch();                                      // in this order: see ln_bwd_kernel
    const size_t off = live ? static_cast<size_t>(row) * d + 8 * lane : 0;
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        const uint32_t dst = smem_u32(mine + 32 * j);
        cp_async_16(dst, dh + off + 256 * j, live);
        cp_async_16(dst + kTensor * 16, x + off + 256 * j, live);
        cp_async_16(dst + 2 * kTensor * 16, resid ? resid + off + 256 * j : dh + off + 256 * j, live && resid != nullptr);   // no residual: zeros
    }
    cp_async_commit();
    const float m = live ? mu[row] : 0.f, r = live ? rstd[row] : 0.f;
    uint4 gm[CH];
#pragma unroll
    for (int j = 0; j < CH; ++j) gm[j] = *reinterpret_cast<const uint4*>(gamma + 8 * lane + 256 * j);
    const uint64_t r2 = splat2(r), nmr2 = splat2(-m * r);
    if (lane == 0) { stats[warp][0] = r; stats[warp][1] = -m * r; }
    cp_async_wait<0>();
    uint64_t s1p = 0ull, s2p = 0ull;
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        uint64_t a[4], b[4], c[4];
        unpack8_pairs(mine[32 * j], a);
        unpack8_pairs(mine[kTensor + 32 * j], b);
        unpack8_pairs(gm[j], c);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint64_t g = fmul2(a[k], c[k]);
            s1p = fadd2(s1p, g);
            s2p = ffma2(g, ffma2(b[k], r2, nmr2), s2p);
        }
    }
    float s1, s1b, s2, s2b;
    unpack_f32x2(s1p, s1, s1b);
    unpack_f32x2(s2p, s2, s2b);
    s1 = warp_sum(s1 + s1b);
    s2 = warp_sum(s2 + s2b);
    const uint64_t nmg2 = splat2(-s1 * (1.0f / d)), nmgx2 = splat2(-s2 * (1.0f / d));
#pragma unroll
    for (int j = 0; j < CH; ++j) {
        uint64_t a[4], b[4], c[4], rs[4];
        unpack8_pairs(mine[32 * j], a);
        unpack8_pairs(mine[kTensor + 32 * j], b);
        unpack8_pairs(mine[2 * kTensor + 32 * j], rs);
        unpack8_pairs(gm[j], c);
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // dx = resid + rstd * (g - mean(g) - xh * mean(g * xh))
            const uint64_t t = ffma2(ffma2(b[k], r2, nmr2), nmgx2, fadd2(fmul2(a[k], c[k]), nmg2));
            w[k] = pack_pair_bf16(ffma2(r2, t, rs[k]));
        }
        const uint4 out = make_uint4(w[0], w[1], w[2], w[3]);
        if (live) *reinterpret_cast<uint4*>(dx + off + 256 * j) = out;
        if (BIAS_SUMS) mine[3 * kTensor + 32 * j] = live ? out : make_uint4(0, 0, 0, 0);    // (0 times an infinite gamma is no zero)
    }
    __syncthreads();
    // columns 4 c .. + 3 of the eight rows
    constexpr int NQ = BIAS_SUMS ? 4 : 2;
    float* prow = partials + static_cast<size_t>(blockIdx.x) * NQ * d;
    const uint2* cols = reinterpret_cast<const uint2*>(ln_rows_smem);
    auto pairs = [](const uint2& v, uint64_t& lo, uint64_t& hi) { lo = pack_f32x2(bf16_lo(v.x), bf16_hi(v.x)); hi = pack_f32x2(bf16_lo(v.y), bf16_hi(v.y)); };
#pragma unroll
    for (int i = 0; i < (d / 4 + 32 * kLnRows - 1) / (32 * kLnRows); ++i) {
        const int c = threadIdx.x + i * 32 * kLnRows;
        if (c >= d / 4) break;
        uint64_t acc[NQ][2] = {};
#pragma unroll
        for (int q = 0; q < kLnRows; ++q) {
            const uint64_t rr = splat2(stats[q][0]), nn = splat2(stats[q][1]);
            uint64_t lo, hi, xlo, xhi;
            pairs(cols[q * (d / 4) + c], lo, hi);
            pairs(cols[2 * kTensor + q * (d / 4) + c], xlo, xhi);
            acc[0][0] = ffma2(lo, ffma2(xlo, rr, nn), acc[0][0]);
            acc[0][1] = ffma2(hi, ffma2(xhi, rr, nn), acc[0][1]);
            acc[1][0] = fadd2(acc[1][0], lo);
            acc[1][1] = fadd2(acc[1][1], hi);
            if constexpr (BIAS_SUMS) {
                pairs(cols[4 * kTensor + q * (d / 4) + c], lo, hi);
                acc[2][0] = fadd2(acc[2][0], lo);
                acc[2][1] = fadd2(acc[2][1], hi);
                // the bias gradient sums the values that are actually stored
                pairs(cols[6 * kTensor + q * (d / 4) + c], lo, hi);
                acc[3][0] = fadd2(acc[3][0], lo);
                acc[3][1] = fadd2(acc[3][1], hi);
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) *reinterpret_cast<ulonglong2*>(prow + q * d + 4 * c) = make_ulonglong2(acc[q][0], acc[q][1]);
    }
}

// out[c] (+)= sum over partial rows r of src[r * stride + c], for up to eight (src, out) entries in one
// launch (grid.y = entry): the partial rows of the two LayerNorm backward kernels and of the two bias
// column sums of a layer's backward end up in one launch.  CTA = 64 columns x 16 row lanes, a thread
// owns four consecutive columns (16-byte loads, eight rows in flight): row lane y adds rows y, y+16, ...
// in order, then the 16 lane sums are added in order, so the result does not depend on scheduling.
// n is a multiple of 4.
struct ReduceEntry { const float* src; float* out; int nrows, n; long long stride; };
struct ReduceTable { ReduceEntry e[kReduceMaxEntries]; };
constexpr int kReduceCols = 64, kReduceLanes = 16;
__global__ void __launch_bounds__(kReduceCols / 4 * kReduceLanes)
reduce_partials_kernel(const __grid_constant__ ReduceTable tab, int accumulate)
{
    __shared__ float4 sm[kReduceLanes][kReduceCols / 4];
    const int cx = threadIdx.x & (kReduceCols / 4 - 1), ry = threadIdx.x / (kReduceCols / 4);
    const int c = blockIdx.x * kReduceCols + cx * 4;
    const ReduceEntry& en = tab.e[blockIdx.y];
    float* out = en.out;
    const int n = en.n, nrows = en.nrows;
    grid_dep_launch();
    grid_dep_wait();
    if (out == nullptr || blockIdx.x * kReduceCols >= n) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < n) {
        const size_t stride = static_cast<size_t>(en.stride);          // floats between partial rows
        const float* src = en.src + c;
        int r = ry;
        for (; r + 7 * kReduceLanes < nrows; r += 8 * kReduceLanes) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = *reinterpret_cast<const float4*>(src + (r + u * kReduceLanes) * stride);
#pragma unroll
            for (int u = 0; u < 8; ++u) { s.x += v[u].x; s.y += v[u].y; s.z += v[u].z; s.w += v[u].w; }
        }
        for (; r < nrows; r += kReduceLanes) {
            const float4 v = *reinterpret_cast<const float4*>(src + r * stride);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
    }
    sm[ry][cx] = s;
    __syncthreads();
    if (ry == 0 && c < n) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < kReduceLanes; ++i) { const float4 v = sm[i][cx]; t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w; }
        if (accumulate) { t.x += out[c]; t.y += out[c + 1]; t.z += out[c + 2]; t.w += out[c + 3]; }
        out[c] = t.x; out[c + 1] = t.y; out[c + 2] = t.z; out[c + 3] = t.w;
    }
}

// Column sums of a bf16 [T, N] matrix: CTA (x, y) owns columns 256 x .. +255 and, eight rows at a time (one per warp), rows
// 8 y + w, 8 (y + R) + w, ...; four rows are in flight per thread.  The eight warps' sums meet in shared memory in warp
// order, so a CTA leaves one partial row whatever its share of the rows.
constexpr int kColsumCols = 256;
__global__ void __launch_bounds__(256)
colsum_kernel(const __nv_bfloat16* in, int T, int N, int ld, float* partials)
{
    __shared__ float4 sm[kMaxWarps][2][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int col = blockIdx.x * kColsumCols + lane * 8;
    grid_dep_launch();
    grid_dep_wait();
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (col < N) {
        const int step = 8 * gridDim.y;
        int t = 8 * blockIdx.y + warp;
        for (; t + 3 * step < T; t += 4 * step) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const uint4*>(in + static_cast<size_t>(t + u * step) * ld + col);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float f[8];
                unpack8(v[u], f);
#pragma unroll
                for (int k = 0; k < 8; ++k) acc[k] += f[k];
            }
        }
        for (; t < T; t += step) {
            float f[8];
            unpack8(*reinterpret_cast<const uint4*>(in + static_cast<size_t>(t) * ld + col), f);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] += f[k];
        }
    }
    sm[warp][0][lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    sm[warp][1][lane] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    __syncthreads();
    if (warp < 2 && col < N) {
        float4 s = sm[0][warp][lane];
#pragma unroll
        for (int w = 1; w < kMaxWarps; ++w) {
            const float4 v = sm[w][warp][lane];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4*>(partials + static_cast<size_t>(blockIdx.y) * N + col + 4 * warp) = s;
    }
}

// The column sums of two bf16 matrices of the same T rows, made to run beside the weight-gradient kernel launched in front:
// that one leaves an SM 512 bytes of shared memory and 40,000 registers, and HBM mostly idle.  So: one CTA per SM, no shared
// memory, and a warp for every (256 columns, share of the rows), which leaves a partial row of its own.  Starts without a wait,
// because the kernel in front does (launch_wgrad, late) and reads the same operands; waits before it ends, so
// that its end implies that kernel's.  __ldcg: nothing that an L1 may still hold from before those operands were written.
// In front of the weight gradients instead, as two launches that shared no SM with them (us for the whole layer): 1024 x 1024
// tokens 171.8 -> 167.9, 1280 wide 283.8 -> 279.4, 8192 x 2048 wide 2385 -> 2356, 8192 x 1024 wide lean 1115 -> 1093.
constexpr int kBesideWarps = 16;
struct ColsumBeside { const __nv_bfloat16* in[2]; float* partials[2]; int n[2]; int T, blocks0, blocks, rows; };
__global__ void __launch_bounds__(32 * kBesideWarps)
colsum_beside_kernel(const ColsumBeside p)
{
    const int lane = threadIdx.x & 31;
    grid_dep_launch();
    const int units = p.blocks * p.rows;
    for (int u = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; u < units; u += kBesideWarps * gridDim.x) {
        const int r = u / p.blocks, blk = u - r * p.blocks, job = blk >= p.blocks0;
        const int N = job ? p.n[1] : p.n[0], col = (blk - (job ? p.blocks0 : 0)) * kColsumCols + lane * 8;
        if (col >= N) continue;
        const __nv_bfloat16* src = (job ? p.in[1] : p.in[0]) + col;
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        int t = r;
        for (; t + 7 * p.rows < p.T; t += 8 * p.rows) {
            uint4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldcg(reinterpret_cast<const uint4*>(src + static_cast<size_t>(t + i * p.rows) * N));
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float f[8];
                unpack8(v[i], f);
#pragma unroll
                for (int k = 0; k < 8; ++k) acc[k] += f[k];
            }
        }
        for (; t < p.T; t += p.rows) {
            float f[8];
            unpack8(__ldcg(reinterpret_cast<const uint4*>(src + static_cast<size_t>(t) * N)), f);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] += f[k];
        }
        float4* dst = reinterpret_cast<float4*>((job ? p.partials[1] : p.partials[0]) + static_cast<size_t>(r) * N + col);
        dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    grid_dep_wait();
}

// Partial rows: as many as the warps of the chip allow, but at least 32 rows of the matrices for each.
int colsum_beside_rows(int sm_count, int T, int N0, int N1)
{
    const int blocks = (N0 + kColsumCols - 1) / kColsumCols + (N1 + kColsumCols - 1) / kColsumCols;
    int r = kBesideWarps * sm_count / blocks;
    if (r > (T + 31) / 32) r = (T + 31) / 32;
    return r < 1 ? 1 : r;
}

// Partial rows: about four CTAs per SM, but at least 32 rows of the matrix for each, so that on few tokens the
// partial rows stay a small part of what they summarise: 1024 x 2048 8.1 -> 3.7 us with the reduce launch, 1024 x 4096
// 6.6 -> 3.8, 8192 x 4096 15.6 -> 14.5 (against one warp-wide row per thread column and up to T partial rows).
int colsum_splits(int sm_count, int T, int N)
{
    const int col_blocks = (N + kColsumCols - 1) / kColsumCols;
    int r = (4 * sm_count + col_blocks - 1) / col_blocks;
    if (r > (T + 31) / 32) r = (T + 31) / 32;
    return r;
}

// Eight rows a CTA while the CTAs are at most some three rounds; beyond, their partial rows (one per CTA, an eighth of the input) and the missing
// overlap of a row's loads with the last one's sums cost more.  us with the reduce launch, persistent -> eight rows: 128 x 256
// 3.9 -> 3.0, 2048 x 256 4.8 -> 4.5, 3072 x 256 5.3 -> 5.7; 1024 x 512 5.6 -> 3.8, 4096 x 512 8.4 -> 8.4, 8192 x 512 13.5 -> 14.3; 512 x 1024
// 5.8 -> 4.2, 1024 x 1024 7.5 -> 4.7, 2368 x 1024 9.8 -> 8.7, 4096 x 1024 13.6 -> 12.2, 8192 x 1024 19.7 -> 20.1; 2048 x 1280 12.6 -> 7.6, 4096 x 1280
// 18.6 -> 14.2, 4096 x 1792 19.6 -> 18.3, 6144 x 1792 25.6 -> 26.1; a row of 2048 leaves one CTA an SM: 512 x 2048 8.6 -> 6.0, 2048 x 2048 15.0 -> 14.0,
// 3072 x 2048 17.9 -> 19.5, and 128 x 2048 5.2 -> 5.7.  Without the two bias sums the lines lie where they do with them: 256 x 2048 5.05 -> 5.15, 512 x 2048
// 6.4 -> 5.7, 2048 x 2048 12.7 -> 12.5, 4096 x 1792 17.3 -> 15.8, 4096 x 1024 12.3 -> 11.3.
bool ln_bwd_by_rows(int T, int d)
{
    return d < 2048 ? T <= (d == 256 ? 2048 : 4096) : d == 2048 && T > 128 && T <= 2048;
}

// Persistent CTAs.  A row slot takes at least four rows, unless that leaves fewer CTAs than keep the loads in flight: 64, or 128 for rows of
// more than 4096, where a CTA has one slot and a row takes longer.  On few tokens the partial rows, one per CTA, then stay a small part
// of the input.  us with the reduce launch, one row / four rows a slot / this: 128 x 6144 11.4 / 12.9 / 11.4, 128 x 8192 14.0 / 16.7 / 13.8,
// 256 x 8192 16.9 / 18.6 / 16.1, 512 x 4096 10.0 / 10.5 / 10.6.
int ln_bwd_grid(Runtime* rt, int T, int d, const RowPlan& rp)
{
    if (ln_bwd_by_rows(T, d)) return (T + kLnRows - 1) / kLnRows;
    const int row_groups = (T + rp.rows_per_cta - 1) / rp.rows_per_cta;
    const int cap = (rp.chunks == 1 ? 2 : 1) * rt->sm_count;
    const int least = rp.chunks == 4 ? std::min(row_groups, 128) : std::min((row_groups + 1) / 2, 64);
    return std::min(std::max((row_groups + 3) / 4, least), cap);
}

}  // namespace

const char* launch_layernorm_fwd(Runtime* rt, const void* x, const void* gamma, const void* beta, int T, int d,
                                 float eps, void* h, void* mu, void* rstd, cudaStream_t stream)
{
    int W = 0, CH = 0;
    if (T <= 0 || !plan_warp_rows(d, &W, &CH)) return "layernorm: unsupported row width";
    const int rows_per_cta = kMaxWarps / W;
    const int grid = (T + rows_per_cta - 1) / rows_per_cta;
    auto X = static_cast<const __nv_bfloat16*>(x);
    auto G = static_cast<const __nv_bfloat16*>(gamma);
    auto Bt = static_cast<const __nv_bfloat16*>(beta);
    auto Hh = static_cast<__nv_bfloat16*>(h);
    auto Mu = static_cast<float*>(mu);
    auto Rs = static_cast<float*>(rstd);
    const bool few = grid <= rt->sm_count;
#define PW_LN_FWD(N) case N: le = few ? launch_k(ln_fwd_kernel<N, true>, dim3(grid), dim3(kRowThreadsMax), 0, stream, X, G, Bt, T, d, eps, Hh, Mu, Rs, W) \
                                      : launch_k(ln_fwd_kernel<N, false>, dim3(grid), dim3(kRowThreadsMax), 0, stream, X, G, Bt, T, d, eps, Hh, Mu, Rs, W); break
    cudaError_t le = cudaSuccess;
    switch (CH) {
        PW_LN_FWD(1); PW_LN_FWD(2); PW_LN_FWD(3); PW_LN_FWD(4); PW_LN_FWD(5); PW_LN_FWD(6); PW_LN_FWD(7); PW_LN_FWD(8);
        default: return "layernorm: unsupported row width";
    }
#undef PW_LN_FWD
    return le == cudaSuccess ? nullptr : "layernorm fwd launch failed";
}

const char* configure_elementwise()
{
    cudaError_t e = cudaSuccess;
#define PW_LN_ATTR(C, B) if (e == cudaSuccess) e = cudaFuncSetAttribute(ln_bwd_kernel<C, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, ln_bwd_depth(C) * 3 * C * kRowThreadsMax * 16)
    PW_LN_ATTR(1, true); PW_LN_ATTR(1, false); PW_LN_ATTR(2, true); PW_LN_ATTR(2, false); PW_LN_ATTR(4, true); PW_LN_ATTR(4, false);
#undef PW_LN_ATTR
#define PW_LN_ATTR(N) if (e == cudaSuccess) e = cudaFuncSetAttribute(ln_bwd_rows_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ln_rows_smem_bytes(N, true)); \
                      if (e == cudaSuccess) e = cudaFuncSetAttribute(ln_bwd_rows_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ln_rows_smem_bytes(N, false))
    PW_LN_ATTR(1); PW_LN_ATTR(2); PW_LN_ATTR(3); PW_LN_ATTR(4); PW_LN_ATTR(5); PW_LN_ATTR(6); PW_LN_ATTR(7); PW_LN_ATTR(8);
#undef PW_LN_ATTR
    return e == cudaSuccess ? nullptr : "could not raise the shared-memory limit of the layernorm kernels";
}

size_t layernorm_bwd_scratch_bytes(Runtime* rt, int T, int d)
{
    RowPlan rp;
    if (T <= 0 || !plan_rows(d, &rp)) return 0;
    return static_cast<size_t>(ln_bwd_grid(rt, T, d, rp)) * 4 * d * sizeof(float);
}

// Main kernel only: the partial rows stay in `partials` and `job` says how to reduce them.
const char* launch_layernorm_bwd_partial(Runtime* rt, const void* dh, const void* x, const void* mu, const void* rstd,
                                         const void* gamma, const void* resid, int T, int d, void* dx, void* dgamma,
                                         void* dbeta, void* db_resid, void* db_dx, void* partials, ReduceJob* job,
                                         cudaStream_t stream)
{
    RowPlan rp;
    if (T <= 0 || !plan_rows(d, &rp)) return "layernorm: unsupported row width";
    const int grid = ln_bwd_grid(rt, T, d, rp);
    auto DH = static_cast<const __nv_bfloat16*>(dh);
    auto X = static_cast<const __nv_bfloat16*>(x);
    auto G = static_cast<const __nv_bfloat16*>(gamma);
    auto R = static_cast<const __nv_bfloat16*>(resid);
    auto DX = static_cast<__nv_bfloat16*>(dx);
    auto Mu = static_cast<const float*>(mu);
    auto Rs = static_cast<const float*>(rstd);
    auto P = static_cast<float*>(partials);
    cudaError_t le = cudaSuccess;
    const bool by_rows = ln_bwd_by_rows(T, d);
    const size_t ring_bytes = static_cast<size_t>(ln_bwd_depth(rp.chunks)) * 3 * rp.chunks * rp.threads * 16;
    const bool sums = db_resid != nullptr || db_dx != nullptr;
#define PW_LN_BWD(C, B) le = launch_k(ln_bwd_kernel<C, B>, dim3(grid), dim3(rp.threads), ring_bytes, stream, DH, X, Mu, Rs, G, R, T, d, DX, P, rp.tpr, rp.rows_per_cta)
#define PW_LN_ROWS(N) case N: le = sums ? launch_k(ln_bwd_rows_kernel<N, true>, dim3(grid), dim3(32 * kLnRows), ln_rows_smem_bytes(N, true), stream, DH, X, Mu, Rs, G, R, T, DX, P) \
                                        : launch_k(ln_bwd_rows_kernel<N, false>, dim3(grid), dim3(32 * kLnRows), ln_rows_smem_bytes(N, false), stream, DH, X, Mu, Rs, G, R, T, DX, P); break
    if (by_rows) {
        switch (d / 256) { PW_LN_ROWS(1); PW_LN_ROWS(2); PW_LN_ROWS(3); PW_LN_ROWS(4); PW_LN_ROWS(5); PW_LN_ROWS(6); PW_LN_ROWS(7); PW_LN_ROWS(8); default: return "layernorm: unsupported row width"; }
    } else switch (rp.chunks) {
        case 1: if (sums) PW_LN_BWD(1, true); else PW_LN_BWD(1, false); break;
        case 2: if (sums) PW_LN_BWD(2, true); else PW_LN_BWD(2, false); break;
        default: if (sums) PW_LN_BWD(4, true); else PW_LN_BWD(4, false); break;
    }
#undef PW_LN_ROWS
#undef PW_LN_BWD
    if (le != cudaSuccess) return "layernorm bwd launch failed";
    job->partials = P; job->nrows = grid; job->nq = sums ? 4 : 2; job->n = d;
    job->out[0] = static_cast<float*>(dgamma); job->out[1] = static_cast<float*>(dbeta);
    job->out[2] = static_cast<float*>(db_resid); job->out[3] = static_cast<float*>(db_dx);
    return nullptr;
}

// One launch for the partial rows of up to four jobs (at most eight output vectors in all).
const char* launch_reduce_jobs(const ReduceJob* jobs, int njobs, int accumulate, cudaStream_t stream)
{
    ReduceTable tab = {};
    int ne = 0, max_n = 0;
    for (int j = 0; j < njobs; ++j)
        for (int q = 0; q < jobs[j].nq; ++q) {
            if (jobs[j].out[q] == nullptr) continue;
            if (ne == kReduceMaxEntries) return "reduce: too many output vectors for one launch";
            ReduceEntry& en = tab.e[ne++];
            en.src = jobs[j].partials + static_cast<size_t>(q) * jobs[j].n;
            en.out = jobs[j].out[q];
            en.nrows = jobs[j].nrows; en.n = jobs[j].n;
            en.stride = static_cast<long long>(jobs[j].nq) * jobs[j].n;
            if (en.n > max_n) max_n = en.n;
        }
    if (ne == 0) return nullptr;
    dim3 rgrid((max_n + kReduceCols - 1) / kReduceCols, ne);
    return launch_k(reduce_partials_kernel, rgrid, dim3(kReduceCols / 4 * kReduceLanes), 0, stream, tab, accumulate) == cudaSuccess
               ? nullptr : "partial-row reduce launch failed";
}

const char* launch_layernorm_bwd(Runtime* rt, const void* dh, const void* x, const void* mu, const void* rstd,
                                 const void* gamma, const void* resid, int T, int d, void* dx, void* dgamma,
                                 void* dbeta, void* db_resid, void* db_dx, int accumulate, void* partials,
                                 cudaStream_t stream)
{
    ReduceJob job;
    const char* e = launch_layernorm_bwd_partial(rt, dh, x, mu, rstd, gamma, resid, T, d, dx, dgamma, dbeta, db_resid, db_dx,
                                                 partials, &job, stream);
    return e ? e : launch_reduce_jobs(&job, 1, accumulate, stream);
}

// y = x * scale + shift on fp32 vectors: the node type of the paper's Figure 2 program (a: x*2,
// b: x+1, c: x/2), used to run that worked example through the dispatch paths.
const char* launch_affine_f32(const void* x, long long n, float scale, float shift, void* y, cudaStream_t stream)
{
    if (n <= 0) return "affine: empty vector";
    const long long blocks = (n + 255) / 256;
    if (blocks > 0x7fffffffll) return "affine: vector too long";
    return launch_k(affine_f32_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, stream, static_cast<const float*>(x), n,
                    scale, shift, static_cast<float*>(y)) == cudaSuccess
               ? nullptr : "affine launch failed";
}

const char* launch_gelu_fwd(Runtime* rt, const void* u, void* a, long long n, int act, cudaStream_t stream)
{
    if (n <= 0 || (n % 8) != 0) return "gelu: element count must be a positive multiple of 8";
    const long long n8 = n / 8;
    long long blocks = (n8 + 255) / 256;
    const long long cap = static_cast<long long>(rt->sm_count) * 16;
    if (blocks > cap) blocks = cap;
    return launch_k(gelu_fwd_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, stream, static_cast<const __nv_bfloat16*>(u),
                    static_cast<__nv_bfloat16*>(a), n8, act) == cudaSuccess
               ? nullptr : "gelu launch failed";
}

size_t colsum_scratch_bytes(Runtime* rt, int T, int N)
{
    if (T <= 0 || N <= 0) return 0;
    return static_cast<size_t>(colsum_splits(rt->sm_count, T, N)) * N * sizeof(float);
}

size_t colsum_beside_scratch_bytes(Runtime* rt, int T, int N0, int N1)
{
    return static_cast<size_t>(colsum_beside_rows(rt->sm_count, T, N0, N1)) * (static_cast<size_t>(N0) + N1) * sizeof(float);
}

const char* launch_colsum_beside(Runtime* rt, const void* const in[2], const int n[2], int T, void* const out[2], void* partials, ReduceJob jobs[2],
                                 cudaStream_t stream)
{
    if (T <= 0 || n[0] <= 0 || n[1] <= 0 || (n[0] % 8) || (n[1] % 8)) return "colsum: N must be a multiple of 8";
    ColsumBeside p;
    p.T = T;
    p.rows = colsum_beside_rows(rt->sm_count, T, n[0], n[1]);
    p.blocks0 = (n[0] + kColsumCols - 1) / kColsumCols;
    p.blocks = p.blocks0 + (n[1] + kColsumCols - 1) / kColsumCols;
    for (int j = 0; j < 2; ++j) {
        p.in[j] = static_cast<const __nv_bfloat16*>(in[j]);
        p.n[j] = n[j];
        p.partials[j] = static_cast<float*>(partials) + (j ? static_cast<size_t>(p.rows) * n[0] : 0);
        jobs[j].partials = p.partials[j]; jobs[j].nrows = p.rows; jobs[j].nq = 1; jobs[j].n = n[j];
        jobs[j].out[0] = static_cast<float*>(out[j]); jobs[j].out[1] = jobs[j].out[2] = jobs[j].out[3] = nullptr;
    }
    const int units = p.blocks * p.rows;
    const int grid = units < rt->sm_count ? units : rt->sm_count;
    return launch_k(colsum_beside_kernel, dim3(grid), dim3(32 * kBesideWarps), 0, stream, p) == cudaSuccess ? nullptr : "colsum launch failed";
}

static const char* launch_colsum_partial(Runtime* rt, const void* in, int T, int N, int ld, void* out, void* partials, ReduceJob* job, cudaStream_t stream)
{
    if (T <= 0 || N <= 0 || (N % 8) || (ld % 8)) return "colsum: N and ld must be multiples of 8";
    const int R = colsum_splits(rt->sm_count, T, N);
    dim3 grid((N + kColsumCols - 1) / kColsumCols, R);
    if (launch_k(colsum_kernel, grid, dim3(256), 0, stream, static_cast<const __nv_bfloat16*>(in), T, N, ld, static_cast<float*>(partials)) != cudaSuccess)
        return "colsum launch failed";
    job->partials = static_cast<const float*>(partials); job->nrows = R; job->nq = 1; job->n = N;
    job->out[0] = static_cast<float*>(out); job->out[1] = job->out[2] = job->out[3] = nullptr;
    return nullptr;
}

const char* launch_colsum(Runtime* rt, const void* in, int T, int N, int ld, void* out, int accumulate,
                          void* partials, cudaStream_t stream)
{
    ReduceJob job;
    const char* e = launch_colsum_partial(rt, in, T, N, ld, out, partials, &job, stream);
    return e ? e : launch_reduce_jobs(&job, 1, accumulate, stream);
}

// ---------------------------------------------------------------------------------------------
// Column sums without any allocation.  Some callers hand this library buffers but cannot create
// device memory themselves while they run - a serving loop that has already given every byte of
// HBM to its pools, a host callback, code running under a framework that forbids allocation at
// that point.  For them the scratch of the column-sum kernel (the per-row-group partial sums)
// lives in this fixed array, which every GPU that loads the library holds until the process
// exits.  All calls share it: two calls that overlap on the GPU race on it, and it keeps the last
// call's partial sums (every slot that a call reads is first written by that same call, so
// nothing needs clearing).
constexpr size_t kStaticScratchFloats = 262144;   // 1 MiB
static __device__ __align__(256) float g_colsum_scratch[kStaticScratchFloats];

namespace {
struct StaticScratch { float* ptr; int sm_count; };
// In host code the array's name is only a handle for the runtime, not a device address: the
// address comes from cudaGetSymbolAddress, asked once per device with that device current.
const char* static_scratch_for_current_device(StaticScratch* out, int* err_kind)
{
    *err_kind = kErrCuda;
    static std::mutex mu;
    static std::map<int, StaticScratch> per_device;
    std::lock_guard<std::mutex> lock(mu);
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return "no CUDA device (cudaGetDevice failed)";
    auto it = per_device.find(dev);
    if (it == per_device.end()) {
        int major = 0, sms = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return "cudaDeviceGetAttribute failed";
        if (major != 10) { *err_kind = kErrDevice; return "device is not compute capability 10.x (sm_100a kernels only, no fallback)"; }
        float* ptr = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_colsum_scratch);
        if (e != cudaSuccess || ptr == nullptr) return "cudaGetSymbolAddress(static scratch) failed";
        it = per_device.emplace(dev, StaticScratch{ptr, sms}).first;
    }
    *out = it->second;
    return nullptr;
}
}  // namespace

size_t colsum_noalloc_max_columns() { return kStaticScratchFloats; }

const char* launch_colsum_noalloc(const void* in, int T, int N, int ld, void* out, int accumulate, cudaStream_t stream,
                                  int* err_kind)
{
    *err_kind = kErrArgument;
    if (T <= 0 || N <= 0 || (N % 8) || (ld % 8) || ld < N) return "colsum: N and ld must be multiples of 8, ld >= N";
    if (static_cast<size_t>(N) > kStaticScratchFloats)
        return "colsum (no-allocation variant): N exceeds the 262144 columns the built-in scratch can hold";
    StaticScratch sc;
    if (const char* e = static_scratch_for_current_device(&sc, err_kind)) return e;
    *err_kind = kErrCuda;
    // as many row groups as the fixed scratch can hold, at most what the allocating variant uses
    const int col_blocks = (N + kColsumCols - 1) / kColsumCols;
    long long R = colsum_splits(sc.sm_count, T, N);
    const long long fit = static_cast<long long>(kStaticScratchFloats / static_cast<size_t>(N));
    if (R > fit) R = fit;
    dim3 grid(col_blocks, static_cast<unsigned>(R));
    colsum_kernel<<<grid, 256, 0, stream>>>(static_cast<const __nv_bfloat16*>(in), T, N, ld, sc.ptr);
    if (cudaGetLastError() != cudaSuccess) return "colsum launch failed";
    ReduceTable tab = {};
    tab.e[0].src = sc.ptr; tab.e[0].out = static_cast<float*>(out);
    tab.e[0].nrows = static_cast<int>(R); tab.e[0].n = N; tab.e[0].stride = N;
    dim3 rgrid((N + kReduceCols - 1) / kReduceCols, 1);
    reduce_partials_kernel<<<rgrid, kReduceCols / 4 * kReduceLanes, 0, stream>>>(tab, accumulate);
    return cudaGetLastError() == cudaSuccess ? nullptr : "colsum reduce launch failed";
}

}  // namespace pw
