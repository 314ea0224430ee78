// head.cu -- the small layers around the convolutions of ResNet-18
// (Sec. 5.1.1): the ImageNet stem's 3x3/2 max pooling, and the head
// (global average pooling -- Sec. 6 -- a fully connected layer and the
// batch-mean softmax cross-entropy of Eq. 1), forward and backward.
//
// These are a few percent of a step's time: the max pool is a bandwidth
// pass over the stem output, the head works on [n, 512] features.  The FC
// products are done by a tiled fp32 GEMM on the CUDA cores.
#include <float.h>

#include <algorithm>
#include <utility>

#include "dbl_internal.cuh"

namespace {

__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8])
{
    const act2_t* h = reinterpret_cast<const act2_t*>(&v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 t = dbl::act::unpack2(h[k]);
        f[2 * k] = t.x;
        f[2 * k + 1] = t.y;
    }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8])
{
    uint4 v;
    act2_t* h = reinterpret_cast<act2_t*>(&v);
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = dbl::act::pack2(f[2 * k], f[2 * k + 1]);
    return v;
}

// Eight floats at a 16-byte aligned address.
__device__ __forceinline__ void load8(const float* p, float (&f)[8])
{
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w;
    f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
}

int grid_for(int64_t items, int threads, int per_sm = 8)
{
    int64_t b = (items + threads - 1) / threads;
    const int64_t cap = (int64_t)dbl::sm_count() * per_sm;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

// ----------------------------------------------------------------------------- max pool 3x3 / 2, pad 1
__global__ void __launch_bounds__(256) maxpool_fwd_kernel(const act_t* __restrict__ x,
                                                          act_t* __restrict__ y, uint8_t* __restrict__ arg,
                                                          int n, int H, int W, int C, int P, int Q)
{
    // 32-bit index math: the host checks that n*P*Q*C/8 fits
    const unsigned groups = (unsigned)C / 8u;
    const unsigned total = (unsigned)n * P * Q * groups;
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const unsigned g = t % groups;
        unsigned pix = t / groups;
        const int q = (int)(pix % (unsigned)Q);
        pix /= (unsigned)Q;
        const int p = (int)(pix % (unsigned)P);
        const int b = (int)(pix / (unsigned)P);
        float best[8];
        uint8_t bi[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            best[k] = -INFINITY;
            bi[k] = 0;
        }
        for (int r = 0; r < 3; ++r) {
            const int h = 2 * p + r - 1;
            if (h < 0 || h >= H) continue;
            for (int s = 0; s < 3; ++s) {
                const int w = 2 * q + s - 1;
                if (w < 0 || w >= W) continue;
                float f[8];
                unpack8(__ldg(reinterpret_cast<const uint4*>(x + (((int64_t)b * H + h) * W + w) * C) + g), f);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (f[k] > best[k]) {  // strict: the first maximum in (r, s) order wins ties
                        best[k] = f[k];
                        bi[k] = (uint8_t)(r * 3 + s);
                    }
            }
        }
        const int64_t o = (((int64_t)b * P + p) * Q + q) * C + 8 * g;
        *reinterpret_cast<uint4*>(y + o) = pack8(best);
        uint2 packed;
        packed.x = bi[0] | (bi[1] << 8) | (bi[2] << 16) | ((uint32_t)bi[3] << 24);
        packed.y = bi[4] | (bi[5] << 8) | (bi[6] << 16) | ((uint32_t)bi[7] << 24);
        *reinterpret_cast<uint2*>(arg + o) = packed;
    }
}

// The same max pool over the output of a training-mode BatchNorm + ReLU
// (no residual) that is never stored: each input vector is normalised as the
// BatchNorm pass would store it, bf16(relu(y*scale + shift)) with the same
// fp32 operations, and then pooled, so the pooled values and the argmax are
// those of pooling the stored BatchNorm output.
// One pair of channels of one input vector through BatchNorm + ReLU, as
// 16-bit pairs of the storage format: each lane is the rounded y*scale + shift from one
// fp32 fma, then max(., 0) in that format, which maps negatives and NaN to zero like the stored
// pass's relu.  A result may be -0 where that pass stores +0; the pool's
// comparisons treat the two alike and the stored maximum is made +0.
__device__ __forceinline__ uint32_t bn_relu_pair(uint32_t w, float2 sc, float2 sh)
{
    const float2 x = dbl::act::unpack2_u32(w);
    const float o0 = __fmaf_rn(x.x, sc.x, sh.x);
    const float o1 = __fmaf_rn(x.y, sc.y, sh.y);
    uint32_t v;
    asm("cvt.rn." DBL_ACT_X2 ".f32 %0, %1, %2;" : "=r"(v) : "f"(o1), "f"(o0));
    asm("max." DBL_ACT_X2 " %0, %1, %2;" : "=r"(v) : "r"(v), "r"(0u));
    return v;
}

// The taps of a window are visited last to first with a >= comparison, so the
// index left is the first maximum in (r, s) order, as in the plain max pool.
// A thread keeps one channel group g for all its windows (the block size is a
// multiple of C/8), so the per-channel scale and shift are computed once, and
// it walks its windows by a fixed pixel stride with carries instead of
// divisions.
__global__ void __launch_bounds__(256)
    bn_relu_maxpool_fwd_kernel(const act_t* __restrict__ x, const float* __restrict__ gamma,
                               const float* __restrict__ beta, const float* __restrict__ mean,
                               const float* __restrict__ invstd, act_t* __restrict__ y,
                               uint8_t* __restrict__ arg, int n, int H, int W, int C, int P, int Q)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    const unsigned groups = (unsigned)C / 8u;
    const unsigned per_block = blockDim.x / groups;
    if (threadIdx.x >= per_block * groups) return;
    const unsigned g = threadIdx.x % groups;
    const unsigned npix = (unsigned)n * P * Q;
    unsigned pix = blockIdx.x * per_block + threadIdx.x / groups;
    const unsigned stride = gridDim.x * per_block;
    int q = (int)(pix % (unsigned)Q), p = (int)((pix / (unsigned)Q) % (unsigned)P),
        b = (int)(pix / ((unsigned)Q * P));
    const int step_q = (int)(stride % (unsigned)Q), step_p = (int)((stride / (unsigned)Q) % (unsigned)P),
              step_b = (int)(stride / ((unsigned)Q * P));
    float2 sc[4], sh[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c0 = 8 * g + 2 * k;
        dbl::dev::bn_scale_shift(gamma[c0], beta[c0], mean[c0], invstd[c0], sc[k].x, sh[k].x);
        dbl::dev::bn_scale_shift(gamma[c0 + 1], beta[c0 + 1], mean[c0 + 1], invstd[c0 + 1], sc[k].y, sh[k].y);
    }
    const int64_t row_vecs = (int64_t)W * groups;  // uint4 vectors per input row
    for (; pix < npix; pix += stride) {
        const uint4* xv = reinterpret_cast<const uint4*>(x) + ((int64_t)b * H + 2 * p - 1) * row_vecs +
                          (int64_t)(2 * q - 1) * groups + g;
        const bool r_ok[3] = {p > 0, true, 2 * p + 1 < H};
        const bool s_ok[3] = {q > 0, true, 2 * q + 1 < W};
        // rows last to first, the next row's loads in flight while one is pooled
        uint32_t best[4] = {0u, 0u, 0u, 0u}, idx[4] = {0u, 0u, 0u, 0u};
        uint4 cur[3], nxt[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            cur[s] = (r_ok[2] && s_ok[s]) ? __ldg(xv + 2 * row_vecs + s * (int64_t)groups) : make_uint4(0u, 0u, 0u, 0u);
            nxt[s] = s_ok[s] ? __ldg(xv + row_vecs + s * (int64_t)groups) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int r = 2; r >= 0; --r) {
            if (r_ok[r]) {
#pragma unroll
                for (int s = 2; s >= 0; --s) {
                    if (!s_ok[s]) continue;
                    const uint32_t tap = (uint32_t)(3 * r + s) * 0x10001u;
                    const uint32_t w[4] = {cur[s].x, cur[s].y, cur[s].z, cur[s].w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t a = bn_relu_pair(w[k], sc[k], sh[k]);
                        uint32_t ge, m;
                        asm("set.ge.u32." DBL_ACT_X2 " %0, %1, %2;" : "=r"(ge) : "r"(a), "r"(best[k]));
                        asm("max." DBL_ACT_X2 " %0, %1, %2;" : "=r"(m) : "r"(best[k]), "r"(a));
                        best[k] = m;
                        idx[k] = (ge & tap) | (~ge & idx[k]);
                    }
                }
            }
            if (r > 0) {
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    cur[s] = nxt[s];
                    if (r == 2)
                        nxt[s] = (r_ok[0] && s_ok[s]) ? __ldg(xv + s * (int64_t)groups) : make_uint4(0u, 0u, 0u, 0u);
                }
            }
        }
        uint4 out;
        // +0 for a maximum of zero (a -0 lane is negative as a signed 16-bit value)
        asm("max.s16x2 %0, %1, %2;" : "=r"(out.x) : "r"(best[0]), "r"(0u));
        asm("max.s16x2 %0, %1, %2;" : "=r"(out.y) : "r"(best[1]), "r"(0u));
        asm("max.s16x2 %0, %1, %2;" : "=r"(out.z) : "r"(best[2]), "r"(0u));
        asm("max.s16x2 %0, %1, %2;" : "=r"(out.w) : "r"(best[3]), "r"(0u));
        const int64_t o = (int64_t)pix * C + 8 * g;
        *reinterpret_cast<uint4*>(y + o) = out;
        *reinterpret_cast<uint2*>(arg + o) = make_uint2(__byte_perm(idx[0], idx[1], 0x6420),
                                                         __byte_perm(idx[2], idx[3], 0x6420));
        q += step_q;
        if (q >= Q) {
            q -= Q;
            ++p;
        }
        p += step_p;
        if (p >= P) {
            p -= P;
            ++b;
        }
        b += step_b;
    }
}

// The same for large tensors (pool_by_rows): a thread owns one channel group g of two neighbouring output columns and walks down `rows` output
// rows: each input row is normalised once, in five vectors of which the middle one serves both columns,
// and reduced along the row (its maximum and the first column that has it); an output row combines three
// such row results, the last of which is the next output row's first.  That is 5 vectors per output
// instead of the 9 of a window taken by itself.  The row maxima combined last row first with >= leave the same
// first maximum.  The five vectors come through a ring of kPoolDepth rows in shared memory that the
// thread fills for itself (cp.async, zeros outside the image): with them in registers, one row ahead, 16 warps
// per SM waited for memory (245 us at 112 x 112 x 64, batch 512, like a window per thread); now 224, 80 x 80 135 -> 120, 144 x 144, batch 185 157 -> 140.
constexpr int kPoolDepth = 5;
// Below this a few long runs of rows leave SMs idle or a last round nearly empty: 64 x 64, batch 64 (34 MB) 15.6 us
// with a window per thread against 16.0 with the best run, 144 x 144, batch 16 (42 MB) 18.4 against 18.3 to 25.9;
// 112 x 112, batch 64 (103 MB) 38.9 against 34.2 to 38.1.
constexpr int64_t kPoolRowsBytes = 96ll << 20;
// With few channels the five columns of a thread's pair are a short run of bytes, and a warp's lie in many lines
// (window per thread and rows, us): 112 x 112, 103 MB: 8 channels 36.8 and 51.3, 16 37.2 and 45.8, 32 36.6 and 39.1; 206 MB: 8 66.7
// and 87.9, 16 66.8 and 76.8, while rows take 65.2 with 32 and 61.7 with 64.  Runs in maps of few rows leave a
// part of their last run empty: 20 x 20, 105 MB, 64 channels 37.2 and 39.7, 256 39.7 and 41.9; 28 x 28 rows 34.0 and 35.9.
constexpr int kPoolRowsMinP = 14;

bool pool_by_rows(int64_t count, int C, int P)
{
    const int64_t bytes = count * C * (int64_t)sizeof(act_t);
    return C >= 32 && P >= kPoolRowsMinP && bytes >= (C >= 64 ? 1 : 2) * kPoolRowsBytes;
}
constexpr int kPoolThreads = 256;

struct PoolRow {  // per column and channel pair: maximum of a row's three taps, and its tap (0..2 in each half)
    uint32_t best[2][4], idx[2][4];
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}

__global__ void __launch_bounds__(kPoolThreads, 2)
    bn_relu_maxpool_rows_kernel(const act_t* __restrict__ x, const float* __restrict__ gamma,
                               const float* __restrict__ beta, const float* __restrict__ mean,
                               const float* __restrict__ invstd, act_t* __restrict__ y,
                               uint8_t* __restrict__ arg, int n, int H, int W, int C, int P, int Q, int rows)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    extern __shared__ uint4 ring[];       // [depth][5][thread]
    const unsigned groups = (unsigned)C / 8u;
    const unsigned per_block = blockDim.x / groups;
    const unsigned g = threadIdx.x % groups;
    const unsigned cols = ((unsigned)Q + 1u) / 2u, chunks = ((unsigned)P + rows - 1u) / rows;
    const unsigned items = (unsigned)n * chunks * cols;
    float2 sc[4], sh[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c0 = 8 * g + 2 * k;
        dbl::dev::bn_scale_shift(gamma[c0], beta[c0], mean[c0], invstd[c0], sc[k].x, sh[k].x);
        dbl::dev::bn_scale_shift(gamma[c0 + 1], beta[c0 + 1], mean[c0 + 1], invstd[c0 + 1], sc[k].y, sh[k].y);
    }
    const int64_t row_vecs = (int64_t)W * groups;  // uint4 vectors per input row
    const uint32_t mine = dbl::dev::smem_u32(ring + threadIdx.x), vec = blockDim.x * 16u;
    for (unsigned item = blockIdx.x * per_block + threadIdx.x / groups; item < items; item += gridDim.x * per_block) {
        const int j = (int)(item % cols), ch = (int)((item / cols) % chunks), b = (int)(item / (cols * chunks));
        const int p0 = ch * rows, p1 = min(P, p0 + rows);
        const int w0 = 4 * j - 1;  // first of the five input columns
        const uint4* xv = reinterpret_cast<const uint4*>(x) + (int64_t)b * H * row_vecs + g;
        bool w_ok[5];
#pragma unroll
        for (int s = 0; s < 5; ++s) w_ok[s] = w0 + s >= 0 && w0 + s < W;
        const int h0 = 2 * p0 - 1, count = 2 * (p1 - p0) + 1;  // input rows h0 .. h0 + count - 1
        auto fetch = [&](int i) {                               // row h0 + i into its slot; always one group
            const int h = h0 + i;
            if (i < count) {
                const bool ok = h >= 0 && h < H;
                const uint32_t dst = mine + (uint32_t)(i % kPoolDepth) * 5u * vec;
#pragma unroll
                for (int s = 0; s < 5; ++s)
                    cp_async16(dst + (uint32_t)s * vec, ok && w_ok[s] ? xv + (int64_t)h * row_vecs + (w0 + s) * (int64_t)groups : xv,
                               ok && w_ok[s]);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // taps outside the image take no part: best starts at zero, and >= against it is only asked of
        // taps inside (every tap is >= 0 after the ReLU, so the last one inside always enters)
        auto reduce_row = [&](int i, PoolRow& row) {
            fetch(i + kPoolDepth - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(kPoolDepth - 1) : "memory");
#pragma unroll
            for (int o = 0; o < 2; ++o)
#pragma unroll
                for (int k = 0; k < 4; ++k) row.best[o][k] = row.idx[o][k] = 0u;
            const uint4* v = ring + threadIdx.x + (i % kPoolDepth) * 5 * blockDim.x;
#pragma unroll
            for (int s = 4; s >= 0; --s) {
                const uint4 t = v[s * blockDim.x];
                if (!w_ok[s]) continue;
                const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t a = bn_relu_pair(w[k], sc[k], sh[k]);
#pragma unroll
                    for (int o = 0; o < 2; ++o) {
                        const int tap = s - 2 * o;
                        if (tap < 0 || tap > 2) continue;
                        uint32_t ge, m;
                        asm("set.ge.u32." DBL_ACT_X2 " %0, %1, %2;" : "=r"(ge) : "r"(a), "r"(row.best[o][k]));
                        asm("max." DBL_ACT_X2 " %0, %1, %2;" : "=r"(m) : "r"(row.best[o][k]), "r"(a));
                        row.best[o][k] = m;
                        row.idx[o][k] = (ge & ((uint32_t)tap * 0x10001u)) | (~ge & row.idx[o][k]);
                    }
                }
            }
        };
#pragma unroll
        for (int i = 0; i < kPoolDepth - 1; ++i) fetch(i);
        PoolRow top;  // row 2p - 1 of the next output row
        reduce_row(0, top);
        for (int p = p0; p < p1; ++p) {
            PoolRow mid, bot;
            reduce_row(2 * (p - p0) + 1, mid);
            reduce_row(2 * (p - p0) + 2, bot);
            const bool top_ok = p > 0, bot_ok = 2 * p + 1 < H;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                if (2 * j + o >= Q) continue;
                uint32_t best[4], idx[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // rows last to first; the middle row is always inside the image
                    uint32_t m = bot.best[o][k], id = bot.idx[o][k] + 0x60006u, ge;
                    if (!bot_ok) m = id = 0u;
                    asm("set.ge.u32." DBL_ACT_X2 " %0, %1, %2;" : "=r"(ge) : "r"(mid.best[o][k]), "r"(m));
                    asm("max." DBL_ACT_X2 " %0, %1, %2;" : "=r"(m) : "r"(m), "r"(mid.best[o][k]));
                    id = (ge & (mid.idx[o][k] + 0x30003u)) | (~ge & id);
                    if (top_ok) {
                        asm("set.ge.u32." DBL_ACT_X2 " %0, %1, %2;" : "=r"(ge) : "r"(top.best[o][k]), "r"(m));
                        asm("max." DBL_ACT_X2 " %0, %1, %2;" : "=r"(m) : "r"(m), "r"(top.best[o][k]));
                        id = (ge & top.idx[o][k]) | (~ge & id);
                    }
                    // +0 for a maximum of zero (a -0 lane is negative as a signed 16-bit value)
                    asm("max.s16x2 %0, %1, %2;" : "=r"(best[k]) : "r"(m), "r"(0u));
                    idx[k] = id;
                }
                const int64_t at = (((int64_t)b * P + p) * Q + 2 * j + o) * C + 8 * g;
                *reinterpret_cast<uint4*>(y + at) = make_uint4(best[0], best[1], best[2], best[3]);
                *reinterpret_cast<uint2*>(arg + at) = make_uint2(__byte_perm(idx[0], idx[1], 0x6420),
                                                                 __byte_perm(idx[2], idx[3], 0x6420));
            }
            top = bot;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");  // the empty groups: counts start anew
    }
}

// a += b, two channels per operation
__device__ __forceinline__ void add8(float (&a)[8], const float (&b)[8])
{
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        const float2 t = dbl::dev::add2(make_float2(a[k], a[k + 1]), make_float2(b[k], b[k + 1]));
        a[k] = t.x, a[k + 1] = t.y;
    }
}

// Gather form over 2x2 blocks of input pixels: block (i, j) = rows 2i..2i+1,
// cols 2j..2j+1 is covered by windows (i..i+1, j..j+1); window (p, q) reaches
// input (h, w) at tap (h - 2p + 1, w - 2q + 1).  So pixel (2i, 2j) takes tap 4
// of window (i, j); (2i, 2j+1) taps 5 and 3 of windows (i, j), (i, j+1);
// (2i+1, 2j) taps 7 and 1 of (i, j), (i+1, j); (2i+1, 2j+1) taps 8, 6, 2, 0
// of the four.  Each pixel sums its windows in (p, q) order, in fp32 from
// zero.  A thread keeps one channel group and steps through the blocks with
// carries, as in the forward pass.  Instruction issue and memory bound it together: the two gradients are
// added two channels per operation, 112x112x64, batch 512 266 -> 242 us, 144x144, batch 185 157.5 -> 147.9 (5.4 TB/s).
__global__ void __launch_bounds__(256)
    maxpool_bwd_kernel(const act_t* __restrict__ dy, const act_t* __restrict__ dy2,
                       const uint8_t* __restrict__ arg, act_t* __restrict__ dx, int n, int H, int W, int C,
                       int P, int Q)
{
    const unsigned groups = (unsigned)C / 8u;
    const unsigned per_block = blockDim.x / groups;
    if (threadIdx.x >= per_block * groups) return;
    const unsigned g = threadIdx.x % groups;
    const int BH = (H + 1) / 2, BW = (W + 1) / 2;  // BH == P and BW == Q
    const unsigned nblk = (unsigned)n * BH * BW;
    unsigned blk = blockIdx.x * per_block + threadIdx.x / groups;
    const unsigned stride = gridDim.x * per_block;
    int j = (int)(blk % (unsigned)BW), i = (int)((blk / (unsigned)BW) % (unsigned)BH),
        b = (int)(blk / ((unsigned)BW * BH));
    const int step_j = (int)(stride % (unsigned)BW), step_i = (int)((stride / (unsigned)BW) % (unsigned)BH),
              step_b = (int)(stride / ((unsigned)BW * BH));
    const int64_t win_row = (int64_t)Q * C;
    for (; blk < nblk; blk += stride) {
        const bool ok[4] = {true, j + 1 < Q, i + 1 < P, i + 1 < P && j + 1 < Q};
        const int64_t o = (((int64_t)b * P + i) * Q + j) * C + 8 * g;  // window (i, j)
        uint4 gv[4], gv2[4];
        uint2 av[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int64_t ot = o + (t >> 1) * win_row + (t & 1) * (int64_t)C;
            gv[t] = ok[t] ? __ldg(reinterpret_cast<const uint4*>(dy + ot)) : make_uint4(0u, 0u, 0u, 0u);
            gv2[t] = (ok[t] && dy2) ? __ldg(reinterpret_cast<const uint4*>(dy2 + ot)) : make_uint4(0u, 0u, 0u, 0u);
            av[t] = ok[t] ? __ldg(reinterpret_cast<const uint2*>(arg + ot)) : make_uint2(~0u, ~0u);
        }
        const bool h1 = 2 * i + 1 < H, w1 = 2 * j + 1 < W;
        act_t* px = dx + (((int64_t)b * H + 2 * i) * W + 2 * j) * C + 8 * g;
        const int64_t px_row = (int64_t)W * C;
        float acc01[8] = {}, acc10[8] = {}, acc11[8] = {};
        {
            float f[8], f2[8], acc00[8] = {};
            unpack8(gv[0], f);
            if (dy2) {
                unpack8(gv2[0], f2);
                add8(f, f2);
            }
            dbl::dev::add_if_tap(acc00, f, av[0], 4);
            dbl::dev::add_if_tap(acc01, f, av[0], 5);
            dbl::dev::add_if_tap(acc10, f, av[0], 7);
            dbl::dev::add_if_tap(acc11, f, av[0], 8);
            *reinterpret_cast<uint4*>(px) = pack8(acc00);
        }
        {
            float f[8], f2[8];
            unpack8(gv[1], f);
            if (dy2) {
                unpack8(gv2[1], f2);
                add8(f, f2);
            }
            dbl::dev::add_if_tap(acc01, f, av[1], 3);
            dbl::dev::add_if_tap(acc11, f, av[1], 6);
            if (w1) *reinterpret_cast<uint4*>(px + C) = pack8(acc01);
        }
        {
            float f[8], f2[8];
            unpack8(gv[2], f);
            if (dy2) {
                unpack8(gv2[2], f2);
                add8(f, f2);
            }
            dbl::dev::add_if_tap(acc10, f, av[2], 1);
            dbl::dev::add_if_tap(acc11, f, av[2], 2);
            if (h1) *reinterpret_cast<uint4*>(px + px_row) = pack8(acc10);
        }
        {
            float f[8], f2[8];
            unpack8(gv[3], f);
            if (dy2) {
                unpack8(gv2[3], f2);
                add8(f, f2);
            }
            dbl::dev::add_if_tap(acc11, f, av[3], 0);
            if (h1 && w1) *reinterpret_cast<uint4*>(px + px_row + C) = pack8(acc11);
        }
        j += step_j;
        if (j >= BW) {
            j -= BW;
            ++i;
        }
        i += step_i;
        if (i >= BH) {
            i -= BH;
            ++b;
        }
        b += step_b;
    }
}

// ----------------------------------------------------------------------------- dropout
// Dropout of the pooled features before the FC layer (Sec. 4.1: the rate rises with the
// resolution, Tables 7 and 9), inverted: a kept feature is scaled by 1/(1 - d).  The draw is
// the counter-based generator Philox4x64-10 (Salmon et al., SC 2011): ten rounds over a
// 256-bit counter with a 128-bit key; a round takes the full 128-bit products of counter
// words 0 and 2 with the two round multipliers and moves the words to
//   (hi(M1*c2) ^ c1 ^ k0, lo(M1*c2), hi(M0*c0) ^ c3 ^ k1, lo(M0*c0)),
// and the key is advanced by the two Weyl increments between rounds.  Feature c of sample n
// takes word c % 4 of the block at counter (n*C/4 + c/4, step, 0, 0), key (seed, 0), and is
// kept when the word's upper 32 bits are >= thr = floor(d * 2^32).
struct Dropout {
    uint32_t thr;          // 0: no dropout
    float scale;           // 1/(1 - d), rounded to fp32
    uint64_t seed;
    const uint64_t* step;  // device counter, read when the kernel runs
    float* mult;           // [n, C] per-feature multiplier (0 or scale) for the backward pass
};

__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1)
{
    constexpr uint64_t kM0 = 0xD2E7470EE14C6C93ull, kM1 = 0xCA5A826395121157ull;
    constexpr uint64_t kW0 = 0x9E3779B97F4A7C15ull, kW1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = kM0 * c[0], q0 = __umul64hi(kM0, c[0]);
        const uint64_t p1 = kM1 * c[2], q1 = __umul64hi(kM1, c[2]);
        const uint64_t a = q1 ^ c[1] ^ k0, b = q0 ^ c[3] ^ k1;
        c[0] = a;
        c[1] = p1;
        c[2] = b;
        c[3] = p0;
        k0 += kW0;
        k1 += kW1;
    }
}

// keep bits (bit j: feature 4*group + j) of one Philox block
__device__ __forceinline__ unsigned dropout_keep4(uint64_t seed, uint64_t step, uint64_t group, uint32_t thr)
{
    uint64_t c[4] = {group, step, 0, 0};
    philox4x64_10(c, seed, 0);
    unsigned bits = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) bits |= (uint32_t)(c[j] >> 32) >= thr ? 1u << j : 0u;
    return bits;
}

__global__ void __launch_bounds__(256) dropout_mask_kernel(int n, int C, uint32_t thr, uint64_t seed,
                                                           const uint64_t* __restrict__ step, uint8_t* __restrict__ keep)
{
    const int64_t groups = (int64_t)n * (C / 4);
    const uint64_t st = thr ? *step : 0;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += (int64_t)gridDim.x * blockDim.x) {
        const unsigned b = thr ? dropout_keep4(seed, st, (uint64_t)g, thr) : 0xFu;
        uchar4 v = make_uchar4(b & 1, (b >> 1) & 1, (b >> 2) & 1, (b >> 3) & 1);
        reinterpret_cast<uchar4*>(keep)[g] = v;
    }
}

// ----------------------------------------------------------------------------- head
// feat[n, c] = mean over hw of x[n, hw, c], then (with dropout) times the feature's multiplier
__global__ void __launch_bounds__(256) avgpool_kernel(const act_t* __restrict__ x, float* __restrict__ feat,
                                                      int n, int hw, int C, Dropout dp)
{
    const int groups = C / 8;
    const int64_t total = (int64_t)n * groups;
    const uint64_t st = dp.thr ? *dp.step : 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(t % groups);
        const int b = (int)(t / groups);
        float acc[8] = {};
        for (int i = 0; i < hw; ++i) {
            float f[8];
            unpack8(__ldg(reinterpret_cast<const uint4*>(x + ((int64_t)b * hw + i) * C) + g), f);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] += f[k];
        }
        const float inv = 1.0f / (float)hw;
        if (dp.thr) {
            const uint64_t q = (uint64_t)b * (uint64_t)(C / 4) + 2 * (uint64_t)g;
            const unsigned bits = dropout_keep4(dp.seed, st, q, dp.thr) | dropout_keep4(dp.seed, st, q + 1, dp.thr) << 4;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float m = (bits >> k) & 1 ? dp.scale : 0.f;
                dp.mult[(int64_t)b * C + 8 * g + k] = m;
                feat[(int64_t)b * C + 8 * g + k] = acc[k] * inv * m;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) feat[(int64_t)b * C + 8 * g + k] = acc[k] * inv;
        }
    }
}

// out[m, n] = sum_k A(m,k) * B(n,k) (+ bias[n]); A(m,k) = A[m*sam + k*sak], B(n,k) = B[n*sbn + k*sbk],
// one of the two strides of each operand being 1.  fp32 on the CUDA cores (the head is fp32 end to
// end): 64 x 128 output tiles, 16-deep K tiles stored K-major in shared memory (double-buffered: the
// next tile is fetched into registers while the current one is multiplied), 8 x 8 outputs per thread,
// two per instruction (fma.rn.f32x2).  The reduction is cut into chunks of kchunk, each a sequential
// fmaf over its k; the chunks of a tile are the CTAs of a cluster (along z), which add their partial
// sums in chunk order through distributed shared memory.  Long reductions of few tiles take several clusters per
// tile (groups), whose sums a second launch adds in order.  Two products, and the loss and bias-gradient
// sums that need the same input, share a launch where that suits both (gemm_plan).
// Bound by fp32 issue: 512 x 1000 x 512 is 7 us of the GPU's fp32 rate.  With 4 x 4 outputs per thread
// (half the FMAs per shared-memory byte), the partial sums through global memory and a launch of their
// own, the head of 512 images and 1000 classes took 128.2 us in ten launches; now 73 in five.
constexpr int GBM = 64, GBN = 128, GBK = 16;
constexpr int GLA = GBM + 4, GLB = GBN + 4;  // row pitches of the K-major tiles
constexpr int kGemmThreads = 128;
constexpr int kGemmMaxCTAs = 608;  // four CTAs per SM of a 152-SM GPU
constexpr int kGemmMaxChunks = 8;  // a cluster

struct GemmJob {
    const float *A, *B, *bias;
    float* out;  // of several groups: their sums [groups][M][N], gstride apart
    int64_t sam, sak, sbn, sbk, ldo, gstride;
    int M, N, K, kchunk, tiles, clusters;  // clusters: tiles x groups
    int vec;  // bits: A, B and out may be accessed 16 bytes at a time
};

// Thread's share of the K tile [k0, k0 + GBK) of rows [row0, row0 + R): float4 number e = tid + 128 q,
// along k or along the rows, whichever is contiguous.
template <int R>
__device__ __forceinline__ void gemm_fetch(const float* __restrict__ X, int64_t s_row, int64_t s_k, bool vec, int row0,
                                           int rows, int k0, int kend, float4 (&t)[R / 32])
{
#pragma unroll
    for (int q = 0; q < R / 32; ++q) {
        const int e = threadIdx.x + kGemmThreads * q;
        const bool along_k = s_k == 1;
        const int row = row0 + (along_k ? e / 4 : e % (R / 4) * 4), k = k0 + (along_k ? e % 4 * 4 : e / (R / 4));
        const float* p = X + (int64_t)row * s_row + (int64_t)k * s_k;
        float f[4];
        if (vec && row + (along_k ? 0 : 3) < rows && k + (along_k ? 3 : 0) < kend) {
            t[q] = __ldg(reinterpret_cast<const float4*>(p));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                f[i] = (row + (along_k ? 0 : i) < rows && k + (along_k ? i : 0) < kend) ? __ldg(p + i) : 0.f;
            t[q] = make_float4(f[0], f[1], f[2], f[3]);
        }
    }
}

template <int R>
__device__ __forceinline__ void gemm_stash(bool along_k, const float4 (&t)[R / 32], float* dst)
{
#pragma unroll
    for (int q = 0; q < R / 32; ++q) {
        const int e = threadIdx.x + kGemmThreads * q;
        if (along_k) {
            float* d = dst + e % 4 * 4 * (R + 4) + e / 4;
            d[0] = t[q].x;
            d[R + 4] = t[q].y;
            d[2 * (R + 4)] = t[q].z;
            d[3 * (R + 4)] = t[q].w;
        } else {
            *reinterpret_cast<float4*>(dst + e / (R / 4) * (R + 4) + e % (R / 4) * 4) = t[q];
        }
    }
}

// What the launch that has dlogits as input also computes (J = 0: nothing): loss = mean(row_loss)
// and db[j] = sum_n dl[n, j].
struct HeadSums {
    const float *row_loss, *dl;
    float *loss, *db;
    int n, J;
};

constexpr int kHeadRedCols = 32;

// Block 0: the loss (256 strided sums, two per thread, then a tree); blocks 1..: 32 columns of db each,
// eight sums of rows w, w + 8, ... in order (two per warp), added in that order.
__device__ __forceinline__ void head_sums(const HeadSums& h, int block, float* red)
{
    const int t = threadIdx.x;
    if (block == 0) {
        float s[2] = {0.f, 0.f};
        for (int i = t; i < h.n; i += 256) {
            s[0] += h.row_loss[i];
            if (i + 128 < h.n) s[1] += h.row_loss[i + 128];
        }
        red[t] = s[0];
        red[t + 128] = s[1];
        __syncthreads();
        for (int w = 128; w; w >>= 1) {
            if (t < w) red[t] += red[t + w];
            __syncthreads();
        }
        if (t == 0) *h.loss = red[0] / (float)h.n;
        return;
    }
    const int lane = t % 32, w = t / 32, j = (block - 1) * kHeadRedCols + lane;
    float s[2] = {0.f, 0.f};
    if (j < h.J) {
#pragma unroll 8
        for (int i = w; i < h.n; i += 8) {
            s[0] += h.dl[(int64_t)i * h.J + j];
            if (i + 4 < h.n) s[1] += h.dl[(int64_t)(i + 4) * h.J + j];
        }
    }
    red[t] = s[0];
    red[t + 128] = s[1];
    __syncthreads();
    if (w == 0 && j < h.J) {
        float v = red[lane];
#pragma unroll
        for (int k = 1; k < 8; ++k) v += red[k * 32 + lane];
        h.db[j] = v;
    }
}

__global__ void __launch_bounds__(kGemmThreads, 4) head_gemm_kernel(const __grid_constant__ GemmJob j0,
                                                                    const __grid_constant__ GemmJob j1,
                                                                    const __grid_constant__ HeadSums hs)
{
    using namespace dbl::dev;
    __shared__ __align__(16) float sm[GBM * GBN];  // K tiles, then the partial sums of this CTA
    static_assert(2 * GBK * (GLA + GLB) <= GBM * GBN, "K tiles");
    const int nz = gridDim.z, z = blockIdx.z;  // the cluster: one CTA per chunk
    int tile = blockIdx.x;
    if (tile >= j0.clusters + j1.clusters) {
        const int b = (tile - j0.clusters - j1.clusters) * nz + z;
        if (b <= (hs.J + kHeadRedCols - 1) / kHeadRedCols) head_sums(hs, b, sm);
        return;
    }
    const GemmJob& j = tile < j0.clusters ? j0 : j1;
    if (tile >= j0.clusters) tile -= j0.clusters;
    int group = 0;
    if (tile >= j.tiles) {
        group = tile / j.tiles;
        tile -= group * j.tiles;
    }
    const int tn = (j.N + GBN - 1) / GBN;
    const int m0 = tile / tn * GBM, n0 = tile % tn * GBN;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;  // rows 4ty.., 32 + 4ty..; columns 4tx.., 64 + 4tx..
    const int kb = (group * nz + z) * j.kchunk, ke = min(j.K, kb + j.kchunk);
    float2 acc[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);
    float4 ra[GBM / 32], rb[GBN / 32];
    gemm_fetch<GBM>(j.A, j.sam, j.sak, j.vec & 1, m0, j.M, kb, ke, ra);
    gemm_fetch<GBN>(j.B, j.sbn, j.sbk, j.vec & 2, n0, j.N, kb, ke, rb);
    float* buf = sm;
    for (int k0 = kb; k0 < ke; k0 += GBK) {
        gemm_stash<GBM>(j.sak == 1, ra, buf);
        gemm_stash<GBN>(j.sbk == 1, rb, buf + GBK * GLA);
        __syncthreads();
        if (k0 + GBK < ke) {  // next tile in flight during the multiply
            gemm_fetch<GBM>(j.A, j.sam, j.sak, j.vec & 1, m0, j.M, k0 + GBK, ke, ra);
            gemm_fetch<GBN>(j.B, j.sbn, j.sbk, j.vec & 2, n0, j.N, k0 + GBK, ke, rb);
        }
        const float *as = buf + 4 * ty, *bs = buf + GBK * GLA + 4 * tx;
#pragma unroll
        for (int k = 0; k < GBK; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(as + k * GLA);
            const float4 a1 = *reinterpret_cast<const float4*>(as + k * GLA + 32);
            const float4 b0 = *reinterpret_cast<const float4*>(bs + k * GLB);
            const float4 b1 = *reinterpret_cast<const float4*>(bs + k * GLB + 64);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 bv[4] = {{b0.x, b0.y}, {b0.z, b0.w}, {b1.x, b1.y}, {b1.z, b1.w}};
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = fma2(make_float2(av[r], av[r]), bv[c], acc[r][c]);
        }
        buf = buf == sm ? sm + GBK * (GLA + GLB) : sm;
    }
    __syncthreads();  // the last tile has been read: sm takes the partial sums
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        float* d = sm + (r / 4 * 32 + 4 * ty + r % 4) * GBN + 4 * tx;
        *reinterpret_cast<float4*>(d) = make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
        *reinterpret_cast<float4*>(d + 64) = make_float4(acc[r][2].x, acc[r][2].y, acc[r][3].x, acc[r][3].y);
    }
    __syncthreads();
    cluster_sync_all();
    // CTA z finishes rows z, z + nz, ... groups of four: 32 threads per row
    const int c = threadIdx.x % 32 * 4, n = n0 + c;
    float bias[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) bias[i] = j.bias && n + i < j.N ? j.bias[n + i] : 0.f;
    for (int r = z * 4 + threadIdx.x / 32; r < GBM; r += 4 * nz) {
        const uint32_t a = smem_u32(sm + r * GBN + c);
        float4 v[kGemmMaxChunks];
#pragma unroll
        for (int q = 0; q < kGemmMaxChunks; ++q)
            if (q < nz) v[q] = ld_cluster_f32x4(mapa_shared(a, (uint32_t)q));
        float4 s = v[0];
#pragma unroll
        for (int q = 1; q < kGemmMaxChunks; ++q)
            if (q < nz) {
                s.x += v[q].x;
                s.y += v[q].y;
                s.z += v[q].z;
                s.w += v[q].w;
            }
        const float o[4] = {s.x + bias[0], s.y + bias[1], s.z + bias[2], s.w + bias[3]};
        const int m = m0 + r;
        if (m < j.M) {
            float* d = j.out + group * j.gstride + (int64_t)m * j.ldo + n;
            if ((j.vec & 4) && n + 3 < j.N) {
                *reinterpret_cast<float4*>(d) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (n + i < j.N) d[i] = o[i];
            }
        }
    }
    cluster_sync_all();  // no CTA leaves while another may still read its partial sums
}

// out[m, n] = the groups' sums part[g][M][N] in order (+ bias[n]).
struct GroupSums {
    const float *part, *bias;
    float* out;
    int64_t ldo;
    int M, N, groups;  // groups = 0: nothing
};

__global__ void __launch_bounds__(256) head_group_reduce_kernel(const __grid_constant__ GroupSums s0,
                                                                const __grid_constant__ GroupSums s1)
{
    for (int x = 0; x < 2; ++x) {
        const GroupSums& s = x ? s1 : s0;
        if (!s.groups) continue;
        const int64_t total = (int64_t)s.M * s.N;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
            float v = s.part[i];
#pragma unroll 8
            for (int g = 1; g < s.groups; ++g) v += s.part[g * total + i];
            const int m = (int)(i / s.N), n = (int)(i % s.N);
            s.out[(int64_t)m * s.ldo + n] = v + (s.bias ? s.bias[n] : 0.f);
        }
    }
}

GemmJob gemm_job(const float* A, int64_t sam, int64_t sak, const float* B, int64_t sbn, int64_t sbk, const float* bias,
                 float* out, int64_t ldo, int M, int N, int K)
{
    GemmJob j{A, B, bias, out, sam, sak, sbn, sbk, ldo, 0, M, N, K, 0, 0, 0, 0};
    auto vec = [](const float* p, int64_t ld) { return dbl::aligned16(p) && ld % 4 == 0; };
    j.vec = (vec(A, sak == 1 ? sam : sak) ? 1 : 0) | (vec(B, sbk == 1 ? sbn : sbk) ? 2 : 0) | (vec(out, ldo) ? 4 : 0);
    return j;
}

// A product as the plan sees it.
struct GemmShape {
    int M, N, K;
    int tiles() const { return ((M + GBM - 1) / GBM) * ((N + GBN - 1) / GBN); }
    // The longest chunk of a product whose result stays fp32: a sum of K terms in few long chains loses more
    // than one in many short ones.  Up to 96 terms cost no more than 64; beyond that enough chunks for about 304
    // tiles of 64 x 64, at least 64 terms each (n images, 10 classes, error of dW against 64 bits with chunks of K / 8
    // and with these: n 1024 9.0e-8 and 6.6e-8, 2048 1.8e-7 and 6.8e-8, 8192 1.3e-6 and 1.0e-7).
    int limit() const
    {
        const int t = ((M + 63) / 64) * ((N + 63) / 64);
        const int z = std::min(std::max((304 + t - 1) / t, 1), std::max(1, (K + 63) / 64));
        return std::max(96, ((K + z - 1) / z + GBK - 1) / GBK * GBK);
    }
};

// How a launch cuts its products' reductions: nz chunks per cluster, groups clusters per tile.
struct GemmPlan {
    int nz, groups[2], kchunk[2];
    double us;  // modelled time
};

// One or two products in a launch.  nz: the most, of 1, 2, 4 and 8, that leaves the longest reduction two K tiles
// per chunk and the grid within the CTAs that are resident at one time.  groups: what the limits ask for, or
// more, for chunks of four K tiles as far as all CTAs are resident, where the model sees a tenth less time.  The model (us):
// 4 for the launch; 1.15 for each K tile of the longest chunk (its loads' latency), or the fp32 rate, 0.54 for each of
// an SM's K tiles; 3 and 3.8 per 1000 CTAs for the exchange; 3 for adding groups.  A function of the shapes only.
GemmPlan gemm_plan(const GemmShape* j, const int* limit, int count)
{
    constexpr int kSMs = kGemmMaxCTAs / 4;
    auto cut = [&](int nz, bool more) {
        GemmPlan p{nz, {1, 1}, {GBK, GBK}, 0.0};
        int tiles = 0, ctas = 0, chain = 0;
        double work = 0.0;
        bool reduce = false;
        for (int i = 0; i < count; ++i) tiles += j[i].tiles();
        for (int i = 0; i < count; ++i) {
            const int K = j[i].K;
            int g = (K + nz * limit[i] - 1) / (nz * limit[i]);
            if (more) g = std::max(g, std::min((K + nz * 4 * GBK - 1) / (nz * 4 * GBK), kGemmMaxCTAs / (tiles * nz)));
            p.kchunk[i] = ((K + nz * g - 1) / (nz * g) + GBK - 1) / GBK * GBK;
            p.groups[i] = (K + nz * p.kchunk[i] - 1) / (nz * p.kchunk[i]);  // none without terms
            ctas += j[i].tiles() * p.groups[i] * nz;
            chain = std::max(chain, p.kchunk[i] / GBK);
            work += (double)j[i].tiles() * ((K + GBK - 1) / GBK);
            reduce = reduce || p.groups[i] > 1;
        }
        p.us = 4.0 + std::max(1.15 * chain, 0.54 / kSMs * work) + (nz > 1 ? 3.0 + 0.0038 * ctas : 0.0) + (reduce ? 3.0 : 0.0);
        return std::make_pair(p, ctas);
    };
    int kmax = 0;
    for (int i = 0; i < count; ++i) kmax = std::max(kmax, j[i].K);
    int nz = 1;
    while (nz < kGemmMaxChunks && kmax >= 2 * nz * 2 * GBK && cut(2 * nz, false).second <= kGemmMaxCTAs) nz *= 2;
    const GemmPlan least = cut(nz, false).first, more = cut(nz, true).first;
    return more.us < 0.9 * least.us ? more : least;
}

// The head's three products.
struct HeadPlan {
    GemmPlan logits, both, dx, dw;
    bool joint;        // df and dW in one launch (both), or one each
    size_t part;       // floats of the groups' sums
};

HeadPlan head_plan(int n, int c, int classes)
{
    const GemmShape f{n, classes, c}, b[2] = {{n, c, classes}, {classes, c, n}};
    // df is rounded to 16 bits
    const int lf = f.limit(), lb[2] = {std::max(256, b[0].limit()), b[1].limit()};
    HeadPlan p;
    p.logits = gemm_plan(&f, &lf, 1);
    p.both = gemm_plan(b, lb, 2);
    p.dx = gemm_plan(&b[0], &lb[0], 1);
    p.dw = gemm_plan(&b[1], &lb[1], 1);
    // Apart, a product of many tiles and few terms does not keep the other from its clusters, at a launch more. The
    // whole head in one launch and so (us): one image of 512 features and 10,000 classes 744 and 70, of 2048 features
    // and 1000 classes 75 and 46, 8192 images of 512 features and 10 classes 735 and 207, 2048 82 and 61.
    // (Where the model sees less than a third between them, one launch measured faster.)
    p.joint = p.both.us <= 1.3 * (p.dx.us + p.dw.us);
    auto part = [](const GemmShape& j, int groups) { return groups > 1 ? (size_t)groups * j.M * j.N : 0; };
    const size_t pb = p.joint ? part(b[0], p.both.groups[0]) + part(b[1], p.both.groups[1])
                              : std::max(part(b[0], p.dx.groups[0]), part(b[1], p.dw.groups[0]));
    p.part = std::max(part(f, p.logits.groups[0]), pb);
    return p;
}

// One or two products (j1 without tiles: none) as plan cuts them, and the sums of hs.
int head_gemm(GemmJob j0, GemmJob j1, const GemmPlan& plan, float* part, const HeadSums& hs, cudaStream_t s,
              const char* what)
{
    GemmJob* job[2] = {&j0, &j1};
    GroupSums groups[2] = {};
    int64_t items = 0;
    for (int i = 0; i < 2; ++i) {
        GemmJob& j = *job[i];
        if (j.M == 0) continue;
        j.tiles = GemmShape{j.M, j.N, j.K}.tiles();
        j.clusters = j.tiles * plan.groups[i];
        j.kchunk = plan.kchunk[i];
        if (plan.groups[i] > 1) {
            groups[i] = {part, j.bias, j.out, j.ldo, j.M, j.N, plan.groups[i]};
            j.gstride = (int64_t)j.M * j.N;
            items = std::max(items, j.gstride);
            j.bias = nullptr;
            j.out = part;
            j.ldo = j.N;
            j.vec = (j.vec & 3) | (dbl::aligned16(part) && j.N % 4 == 0 ? 4 : 0);
            part += plan.groups[i] * j.gstride;
        }
    }
    const int nz = plan.nz;
    const int sums = hs.J ? 1 + (hs.J + kHeadRedCols - 1) / kHeadRedCols : 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = nz;
    cfg.gridDim = dim3(j0.clusters + j1.clusters + (sums + nz - 1) / nz, 1, nz);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, head_gemm_kernel, j0, j1, hs);
    if (e != cudaSuccess) {
        dbl::count_launch();
        return dbl::cuda_check(e, what);
    }
    int rc = dbl::launch_check(what);
    if (rc || !items) return rc;
    head_group_reduce_kernel<<<grid_for(items, 256), 256, 0, s>>>(groups[0], groups[1]);
    return dbl::launch_check(what);
}

// One CTA per row: loss_n = logsumexp(l) - l[label]; dl = (softmax - onehot) * S/n (in place), S the
// loss scale (1 without loss scaling).  (One warp per row, eight rows per CTA, left 88 SMs idle at
// 512 rows and walked 1000 classes in 32 dependent steps per pass.)
constexpr int kSoftmaxThreads = 128;
__global__ void __launch_bounds__(kSoftmaxThreads) softmax_ce_kernel(float* __restrict__ logits,
                                                                     const int32_t* __restrict__ labels, int n, int J,
                                                                     float* __restrict__ row_loss,
                                                                     const float* __restrict__ loss_scale)
{
    __shared__ float red[2][kSoftmaxThreads / 32];
    const int row = blockIdx.x, t = threadIdx.x, w = t / 32;
    float* l = logits + (int64_t)row * J;
    const int lab = labels[row];
    const float invn = (loss_scale ? *loss_scale : 1.0f) / (float)n;
    float mx = -FLT_MAX;
#pragma unroll 8
    for (int j = t; j < J; j += kSoftmaxThreads) mx = fmaxf(mx, l[j]);
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (t % 32 == 0) red[0][w] = mx;
    __syncthreads();
    mx = fmaxf(fmaxf(red[0][0], red[0][1]), fmaxf(red[0][2], red[0][3]));
    float z = 0.f;
#pragma unroll 8
    for (int j = t; j < J; j += kSoftmaxThreads) z += expf(l[j] - mx);
#pragma unroll
    for (int o = 16; o; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if (t % 32 == 0) red[1][w] = z;
    __syncthreads();
    z = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
    const float lse = mx + logf(z);
    if (t == 0) row_loss[row] = lse - l[lab];
    __syncthreads();  // l[lab] has been read
#pragma unroll 8
    for (int j = t; j < J; j += kSoftmaxThreads) l[j] = (expf(l[j] - lse) - (j == lab ? 1.f : 0.f)) * invn;
}

// The same two passes with one CTA per image, blockDim = S slices x (C/8) channel groups: thread
// (slice s, group g) takes the rows i = s, s + S, ... of its image (consecutive threads on
// consecutive 16-byte vectors of a row).  Forward: each slice adds its rows in order, then the S
// slice sums are added in slice order.  Backward: each thread computes its 8 gradients once and
// writes them to its rows.  (One thread per (image, group) walking all hw rows, or loading its
// 16 fp32 factors again for every row, left these passes at a fifth of HBM.)
__device__ __forceinline__ int pool_slices(int groups) { return groups >= 1024 ? 1 : min(8, 1024 / groups); }

__global__ void __launch_bounds__(1024) avgpool_img_kernel(const act_t* __restrict__ x, float* __restrict__ feat,
                                                           int hw, int C, Dropout dp)
{
    extern __shared__ float slice_sum[];  // [S][C], then the keep bits of the C / 4 dropout blocks
    const int groups = C / 8, S = pool_slices(groups);
    uint8_t* keep = reinterpret_cast<uint8_t*>(slice_sum + S * C);
    const int g = threadIdx.x % groups, sl = threadIdx.x / groups;
    const int b = blockIdx.x;
    // the draws first, a block per thread: their long chain of 64-bit products overlaps the other warps' loads
    if (dp.thr) {
        const uint64_t st = *dp.step;
        for (int q = threadIdx.x; q < C / 4; q += blockDim.x)
            keep[q] = (uint8_t)dropout_keep4(dp.seed, st, (uint64_t)b * (uint64_t)(C / 4) + q, dp.thr);
    }
    float acc[8] = {};
#pragma unroll 4
    for (int i = sl; i < hw; i += S) {
        float f[8];
        unpack8(__ldg(reinterpret_cast<const uint4*>(x + ((int64_t)b * hw + i) * C) + g), f);
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] += f[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) slice_sum[sl * C + 8 * g + k] = acc[k];
    __syncthreads();
    // one feature per thread: its slices in order (consecutive threads on consecutive features)
    const float inv = 1.0f / (float)hw;
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        float t = slice_sum[c];
        for (int q = 1; q < S; ++q) t += slice_sum[q * C + c];
        if (dp.thr) {
            const float m = (keep[c / 4] >> (c % 4)) & 1 ? dp.scale : 0.f;
            dp.mult[(int64_t)b * C + c] = m;
            feat[(int64_t)b * C + c] = t * inv * m;
        } else {
            feat[(int64_t)b * C + c] = t * inv;
        }
    }
}

// step (or nullptr): the dropout step counter, advanced once here so that the next call draws a
// fresh mask (every read of it in this call has happened in the forward pool)
__global__ void __launch_bounds__(1024) avgpool_bwd_img_kernel(const float* __restrict__ df, act_t* __restrict__ dx,
                                                               int hw, int C, const float* __restrict__ mult,
                                                               uint64_t* __restrict__ step)
{
    if (step && blockIdx.x == 0 && threadIdx.x == 0) *step += 1;
    const int groups = C / 8, S = pool_slices(groups);
    const int g = threadIdx.x % groups, sl = threadIdx.x / groups;
    const int b = blockIdx.x;
    const float inv = 1.0f / (float)hw;
    float f[8];
    load8(df + (int64_t)b * C + 8 * g, f);
    if (mult) {
        float m[8];
        load8(mult + (int64_t)b * C + 8 * g, m);
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] *= m[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] *= inv;
    const uint4 v = pack8(f);
    uint4* row = reinterpret_cast<uint4*>(dx + (int64_t)b * hw * C) + g;
    for (int i = sl; i < hw; i += S) row[(int64_t)i * groups] = v;
}

// dx[n, i, c] = df[n, c] / hw, with dropout (df[n, c] * mult[n, c]) / hw
__global__ void __launch_bounds__(256) avgpool_bwd_kernel(const float* __restrict__ df, act_t* __restrict__ dx,
                                                          int n, int hw, int C, const float* __restrict__ mult,
                                                          uint64_t* __restrict__ step)
{
    if (step && blockIdx.x == 0 && threadIdx.x == 0) *step += 1;  // as in avgpool_bwd_img_kernel
    const int groups = C / 8;
    const int64_t total = (int64_t)n * hw * groups;
    const float inv = 1.0f / (float)hw;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(t % groups);
        const int b = (int)(t / groups / hw);
        float f[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int64_t e = (int64_t)b * C + 8 * g + k;
            f[k] = (mult ? df[e] * mult[e] : df[e]) * inv;
        }
        reinterpret_cast<uint4*>(dx)[t] = pack8(f);
    }
}

}  // namespace

extern "C" {

int dbl_maxpool_fwd(int32_t n, int32_t h, int32_t w, int32_t c, const void* x, void* y, uint8_t* argmax, void* stream)
{
    using namespace dbl;
    if (n < 0 || h <= 0 || w <= 0 || c <= 0 || !x || !y || !argmax)
        return set_error(DBL_ERR_INVALID, "maxpool_fwd: bad arguments");
    if (c % 8) return set_error(DBL_ERR_INVALID, "maxpool_fwd: channels must be a multiple of 8");
    if (!aligned16(x) || !aligned16(y) || (reinterpret_cast<uintptr_t>(argmax) & 7))
        return set_error(DBL_ERR_INVALID, "maxpool_fwd: misaligned pointer");
    const int P = (h + 2 - 3) / 2 + 1, Q = (w + 2 - 3) / 2 + 1;
    if ((int64_t)n * h * w * (c / 8) >= (int64_t)1 << 31)
        return set_error(DBL_ERR_UNSUPPORTED, "maxpool_fwd: tensor too large for 32-bit indexing");
    if (n == 0) return DBL_OK;
    maxpool_fwd_kernel<<<grid_for((int64_t)n * P * Q * (c / 8), 256), 256, 0, as_stream(stream)>>>(
        static_cast<const act_t*>(x), static_cast<act_t*>(y), argmax, n, h, w, c, P, Q);
    return launch_check("maxpool_fwd launch");
}

int dbl_bn_relu_maxpool_fwd(const dbl_bn_shape* s, int32_t n, int32_t h, int32_t w, const void* x,
                            const float* ch_sum, const float* ch_sumsq, const float* gamma, const float* beta,
                            float* save_mean, float* save_invstd, void* y, uint8_t* argmax, void* stream)
{
    using namespace dbl;
    if (!s || n <= 0 || h <= 0 || w <= 0 || !x || !y || !argmax || !ch_sum || !ch_sumsq || !gamma || !beta ||
        !save_mean || !save_invstd)
        return set_error(DBL_ERR_INVALID, "bn_relu_maxpool_fwd: bad arguments");
    const int c = s->c;
    if (c <= 0 || c % 8 || !s->relu || s->count != (int64_t)n * h * w)
        return set_error(DBL_ERR_INVALID, "bn_relu_maxpool_fwd: shape must be [n*h*w, c], c a multiple of 8, relu set");
    if (c > 8192) return set_error(DBL_ERR_UNSUPPORTED, "bn_relu_maxpool_fwd: at most 8192 channels");
    if (!aligned16(x) || !aligned16(y) || (reinterpret_cast<uintptr_t>(argmax) & 7))
        return set_error(DBL_ERR_INVALID, "bn_relu_maxpool_fwd: misaligned pointer");
    const int P = (h + 2 - 3) / 2 + 1, Q = (w + 2 - 3) / 2 + 1;
    if ((int64_t)n * h * w * (c / 8) >= (int64_t)1 << 31)
        return set_error(DBL_ERR_UNSUPPORTED, "bn_relu_maxpool_fwd: tensor too large for 32-bit indexing");
    cudaStream_t st = as_stream(stream);
    int rc = bn_fwd_finalize(s->count, c, s->eps, ch_sum, ch_sumsq, save_mean, save_invstd, st);
    if (rc) return rc;
    // a block size that is a multiple of the channel groups: each thread keeps its group
    const int groups = c / 8, block = groups * std::max(1, kPoolThreads / groups);
    if (!pool_by_rows(s->count, c, P) || block > kPoolThreads) {
        bn_relu_maxpool_fwd_kernel<<<grid_for((int64_t)n * P * Q, block / groups), block, 0, st>>>(
            static_cast<const act_t*>(x), gamma, beta, save_mean, save_invstd, static_cast<act_t*>(y),
            argmax, n, h, w, c, P, Q);
        return launch_check("bn_relu_maxpool_fwd launch");
    }
    // output rows per thread: the count of two to eight with the least modelled time, rounds of two CTAs per SM
    // (between fractional and whole) x (input rows of a run + ~5 of set-up)
    const int cols = (Q + 1) / 2;
    int rows = 2;
    double best = 0.0;
    for (int r = 2; r <= 8; ++r) {
        const double ctas = (double)n * ((P + r - 1) / r) * cols * groups / kPoolThreads;
        const double waves = std::max(1.0, ctas / (2.0 * sm_count()));
        const double cost = (0.3 * waves + 0.7 * ceil(waves)) * (2 * r + 6);
        if (r == 2 || cost < best) {
            best = cost;
            rows = r;
        }
    }
    const int64_t items = (int64_t)n * ((P + rows - 1) / rows) * cols;
    const size_t smem = (size_t)kPoolDepth * 5 * block * 16;
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        if ((rc = cuda_check(cudaFuncSetAttribute(bn_relu_maxpool_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  kPoolDepth * 5 * kPoolThreads * 16),
                             "bn_relu_maxpool_fwd: set smem attribute")))
            return rc;
        attr_set[dev] = true;
    }
    bn_relu_maxpool_rows_kernel<<<grid_for(items, block / groups), block, smem, st>>>(
        static_cast<const act_t*>(x), gamma, beta, save_mean, save_invstd, static_cast<act_t*>(y),
        argmax, n, h, w, c, P, Q, rows);
    return launch_check("bn_relu_maxpool_fwd launch");
}

int dbl_maxpool_bwd(int32_t n, int32_t h, int32_t w, int32_t c, const void* dy, const void* dy2,
                    const uint8_t* argmax, void* dx, void* stream)
{
    using namespace dbl;
    if (n < 0 || h <= 0 || w <= 0 || c <= 0 || !dy || !dx || !argmax)
        return set_error(DBL_ERR_INVALID, "maxpool_bwd: bad arguments");
    if (c % 8) return set_error(DBL_ERR_INVALID, "maxpool_bwd: channels must be a multiple of 8");
    if (!aligned16(dy) || !aligned16(dx) || (dy2 && !aligned16(dy2)) || (reinterpret_cast<uintptr_t>(argmax) & 7))
        return set_error(DBL_ERR_INVALID, "maxpool_bwd: misaligned pointer");
    const int P = (h + 2 - 3) / 2 + 1, Q = (w + 2 - 3) / 2 + 1;
    if ((int64_t)n * h * w * (c / 8) >= (int64_t)1 << 31)
        return set_error(DBL_ERR_UNSUPPORTED, "maxpool_bwd: tensor too large for 32-bit indexing");
    if (n == 0) return DBL_OK;
    if (c > 8192) return set_error(DBL_ERR_UNSUPPORTED, "maxpool_bwd: at most 8192 channels");
    // a block size that is a multiple of the channel groups: each thread keeps its group
    const int groups = c / 8, block = groups * std::max(1, 256 / groups);
    maxpool_bwd_kernel<<<grid_for((int64_t)n * ((h + 1) / 2) * ((w + 1) / 2), block / groups), block, 0,
                         as_stream(stream)>>>(
        static_cast<const act_t*>(dy), static_cast<const act_t*>(dy2), argmax,
        static_cast<act_t*>(dx), n, h, w, c, P, Q);
    return launch_check("maxpool_bwd launch");
}

size_t dbl_head_workspace_bytes(int32_t n, int32_t c, int32_t classes)
{
    if (n <= 0 || c <= 0 || classes <= 0) return 0;
    // feat, df and the dropout multipliers [n,c], logits/dlogits [n,classes], row_loss [n], then the groups' sums
    const size_t f = (size_t)n * c * 3 + (size_t)n * classes + (size_t)n;
    return (((f + 3) / 4 * 4 + head_plan(n, c, classes).part) * sizeof(float) + 16 + 255) / 256 * 256;  // 16: alignment of the caller's pointer
}

}  // extern "C"

namespace {

int head_fwd_bwd(int32_t n, int32_t hw, int32_t c, int32_t classes, const void* x, const float* fc_w, const float* fc_b,
                 const int32_t* labels, float drop_rate, uint64_t seed, uint64_t* step, const float* loss_scale,
                 float* loss, float* dfc_w, float* dfc_b, void* dx, void* ws, size_t ws_bytes, void* stream,
                 const char* name)
{
    using namespace dbl;
    if (n <= 0 || hw <= 0 || c <= 0 || classes <= 0 || !x || !fc_w || !fc_b || !labels || !loss || !dfc_w || !dfc_b ||
        !dx)
        return set_error(DBL_ERR_INVALID, "%s: bad arguments", name);
    if (c % 8 || !aligned16(x) || !aligned16(dx))
        return set_error(DBL_ERR_INVALID, "%s: channels must be a multiple of 8, tensors 16-byte aligned", name);
    if (!(drop_rate >= 0.f && drop_rate < 1.f))
        return set_error(DBL_ERR_INVALID, "%s: dropout rate %g outside [0, 1)", name, (double)drop_rate);
    if (drop_rate > 0.f && (!step || (reinterpret_cast<uintptr_t>(step) & 7)))
        return set_error(DBL_ERR_INVALID, "%s: dropout needs an 8-byte aligned device step counter", name);
    const size_t need = dbl_head_workspace_bytes(n, c, classes);
    if (!ws || ws_bytes < need) return set_error(DBL_ERR_WORKSPACE, "%s: workspace %zu < %zu", name, ws_bytes, need);
    // c is a multiple of 8, so feat, df, mult and logits are all 16-byte aligned
    float* feat = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(ws) + 15) / 16 * 16);
    float* df = feat + (size_t)n * c;
    float* mult = df + (size_t)n * c;
    float* logits = mult + (size_t)n * c;
    float* row_loss = logits + (size_t)n * classes;
    float* part = feat + ((size_t)n * c * 3 + (size_t)n * classes + (size_t)n + 3) / 4 * 4;
    const HeadPlan plan = head_plan(n, c, classes);
    Dropout dp{0u, 1.f, seed, step, mult};
    if (drop_rate > 0.f) {
        dp.thr = (uint32_t)floor((double)drop_rate * 4294967296.0);
        dp.scale = (float)(1.0 / (1.0 - (double)drop_rate));
    }
    cudaStream_t s = as_stream(stream);
    int rc;
    const int groups = c / 8;
    const bool per_image = groups <= 1024;  // one CTA per image (at most 1024 threads)
    const int S = groups >= 1024 ? 1 : std::min(8, 1024 / groups);
    if (per_image)
        avgpool_img_kernel<<<n, S * groups, (size_t)S * c * sizeof(float) + c / 4, s>>>(static_cast<const act_t*>(x), feat,
                                                                                 hw, c, dp);
    else
        avgpool_kernel<<<grid_for((int64_t)n * groups, 256), 256, 0, s>>>(static_cast<const act_t*>(x), feat, n, hw,
                                                                           c, dp);
    if ((rc = launch_check("avgpool launch"))) return rc;
    // logits = feat * W^T + b
    if ((rc = head_gemm(gemm_job(feat, c, 1, fc_w, c, 1, fc_b, logits, classes, n, classes, c), GemmJob{}, plan.logits,
                        part, HeadSums{}, s, "fc fwd launch")))
        return rc;
    softmax_ce_kernel<<<n, kSoftmaxThreads, 0, s>>>(logits, labels, n, classes, row_loss, loss_scale);
    if ((rc = launch_check("softmax_ce launch"))) return rc;
    // df[n, c] = sum_j dl[n, j] W[j, c]; dW[j, c] = sum_n dl[n, j] feat[n, c]; the loss and db
    const GemmJob jx = gemm_job(logits, classes, 1, fc_w, 1, c, nullptr, df, c, n, c, classes);
    const GemmJob jw = gemm_job(logits, 1, classes, feat, 1, c, nullptr, dfc_w, c, classes, c, n);
    const HeadSums sums{row_loss, logits, loss, dfc_b, n, classes};
    if (plan.joint) {
        if ((rc = head_gemm(jx, jw, plan.both, part, sums, s, "fc bwd launch"))) return rc;
    } else {
        if ((rc = head_gemm(jx, GemmJob{}, plan.dx, part, HeadSums{}, s, "fc dX launch"))) return rc;
        if ((rc = head_gemm(jw, GemmJob{}, plan.dw, part, sums, s, "fc dW launch"))) return rc;
    }
    // with dropout, the pool's backward also advances the step counter (the next call draws a fresh mask)
    uint64_t* adv = dp.thr ? step : nullptr;
    if (per_image)
        avgpool_bwd_img_kernel<<<n, S * groups, 0, s>>>(df, static_cast<act_t*>(dx), hw, c, dp.thr ? mult : nullptr,
                                                        adv);
    else
        avgpool_bwd_kernel<<<grid_for((int64_t)n * hw * groups, 256), 256, 0, s>>>(df, static_cast<act_t*>(dx), n, hw,
                                                                                    c, dp.thr ? mult : nullptr, adv);
    return launch_check("avgpool_bwd launch");
}

}  // namespace

extern "C" {

int dbl_head_fwd_bwd(int32_t n, int32_t hw, int32_t c, int32_t classes, const void* x, const float* fc_w,
                     const float* fc_b, const int32_t* labels, float* loss, float* dfc_w, float* dfc_b, void* dx,
                     void* ws, size_t ws_bytes, void* stream)
{
    return head_fwd_bwd(n, hw, c, classes, x, fc_w, fc_b, labels, 0.f, 0, nullptr, nullptr, loss, dfc_w, dfc_b, dx, ws,
                        ws_bytes, stream, "head_fwd_bwd");
}

int dbl_head_fwd_bwd_ex(int32_t n, int32_t hw, int32_t c, int32_t classes, const void* x, const float* fc_w,
                        const float* fc_b, const int32_t* labels, const dbl_head_opts* opts, float* loss, float* dfc_w,
                        float* dfc_b, void* dx, void* ws, size_t ws_bytes, void* stream)
{
    if (!opts) return dbl::set_error(DBL_ERR_INVALID, "head_fwd_bwd_ex: null options");
    return head_fwd_bwd(n, hw, c, classes, x, fc_w, fc_b, labels, opts->drop_rate, opts->seed, opts->step,
                        opts->loss_scale, loss, dfc_w, dfc_b, dx, ws, ws_bytes, stream, "head_fwd_bwd_ex");
}

int dbl_dropout_mask(int32_t n, int32_t c, float drop_rate, uint64_t seed, const uint64_t* step, uint8_t* keep,
                     void* stream)
{
    using namespace dbl;
    if (n < 0 || c <= 0 || c % 4 || !keep || (reinterpret_cast<uintptr_t>(keep) & 3))
        return set_error(DBL_ERR_INVALID, "dropout_mask: bad arguments (c a multiple of 4, keep 4-byte aligned)");
    if (!(drop_rate >= 0.f && drop_rate < 1.f))
        return set_error(DBL_ERR_INVALID, "dropout_mask: rate %g outside [0, 1)", (double)drop_rate);
    const uint32_t thr = drop_rate > 0.f ? (uint32_t)floor((double)drop_rate * 4294967296.0) : 0u;
    if (thr && (!step || (reinterpret_cast<uintptr_t>(step) & 7)))
        return set_error(DBL_ERR_INVALID, "dropout_mask: needs an 8-byte aligned device step counter");
    if (n == 0) return DBL_OK;
    dropout_mask_kernel<<<grid_for((int64_t)n * (c / 4), 256), 256, 0, as_stream(stream)>>>(n, c, thr, seed, step, keep);
    return launch_check("dropout_mask launch");
}

}  // extern "C"
