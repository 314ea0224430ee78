// bn.cu -- training-mode BatchNorm + residual + ReLU, forward and backward,
// for the ResNet-18 of Sec. 5.1.1.  All kernels are HBM-bound streaming
// passes over [count, C] bf16 tensors with 16-byte (8-channel) vectors.
//
// Forward (one pass, 6 B/element with a residual): the batch statistics come
// from the convolution epilogue (or dbl_bn_stats); every CTA turns them into
// per-channel scale/shift in shared memory, then
//     out = ReLU(y*scale + shift [+ res]).
// Backward (two passes): a reduce pass of sum(g) and sum(g*xhat) per channel
// into per-CTA partials, a tiny fixed-order finalize, and an apply pass
//     dy = gamma*invstd*(g - sum(g)/count - xhat*sum(g*xhat)/count).
#include <algorithm>
#include <mutex>

#include "dbl_internal.cuh"

namespace {

using dbl::dev::bn_scale_shift;

constexpr int kThreads = 256;
constexpr int kMaxC = 2048;
constexpr int kUnroll = 2;  // rows per thread whose loads are in flight together
constexpr int kBlocksPerSM = 4;     // forward apply: 256-thread CTAs resident per SM (64 registers per thread)
constexpr int kBwdBlocksPerSM = 3;  // backward apply pass (85 registers per thread)
constexpr int kReduceBlocksPerSM = 2;  // backward reduce pass: four rows' loads in flight per thread
constexpr int kReduceUnroll = 4;
// Forward apply of tensors above this size: last row first.  The convolution before it wrote y from
// row 0 on, so the end of y is still in L2 when the pass starts, and the pass leaves the first rows of
// out there for the next convolution, which starts at row 0.  Two convolutions and their passes
// (a residual block) against row order: 206 MB and 103 MB tensors 401 -> 394 and 217 -> 210 us, 103 MB
// at 128 channels 267 -> 260 us; at 51 MB, where everything between two passes fits in L2 anyway,
// 143.1 -> 145.5 us and 116.6 -> 118.9 us, so those stay in row order.
constexpr int64_t kReverseAboveBytes = 64ll << 20;

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

// Per-channel constants go to shared memory once per CTA (coalesced) and from there to each thread's
// registers as two 16-byte loads: loading a thread's eight channels from global memory one by one puts
// a warp's 32-byte strides through eight L1 wavefronts per load, 256 of them for the forward apply's
// four arrays, more than the rows of a small tensor cost.  4096
// rows of 512 channels: forward 11.1 -> 8.1 us, backward 18.2 -> 14.7; 25,088 rows 16.3 -> 13.3 and
// 35.0 -> 31.1; 73,728 rows of 128 13.0 -> 11.7 and 26.5 -> 24.9.
__device__ __forceinline__ void load8(const float* s, float (&f)[8])
{
    const float4 a = reinterpret_cast<const float4*>(s)[0], b = reinterpret_cast<const float4*>(s)[1];
    f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w;
    f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
}

// ----------------------------------------------------------------------------- statistics
__global__ void __launch_bounds__(kThreads) bn_stats_kernel(const act_t* __restrict__ y, int64_t count, int C,
                                                            float* __restrict__ sum, float* __restrict__ sumsq)
{
    const int groups = C / 8;
    const int g = threadIdx.x % groups;
    const int rstep = kThreads / groups;
    float s[8] = {}, q[8] = {};
    for (int64_t r = (int64_t)blockIdx.x * rstep + threadIdx.x / groups; r < count; r += (int64_t)gridDim.x * rstep) {
        float f[8];
        unpack8(__ldg(reinterpret_cast<const uint4*>(y + r * C) + g), f);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            s[k] += f[k];
            q[k] = fmaf(f[k], f[k], q[k]);
        }
    }
    __shared__ float red[kThreads][17];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        red[threadIdx.x][k] = s[k];
        red[threadIdx.x][8 + k] = q[k];
    }
    __syncthreads();
    if (threadIdx.x < groups) {
        float ts[8] = {}, tq[8] = {};
        for (int t = threadIdx.x; t < rstep * groups; t += groups)
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                ts[k] += red[t][k];
                tq[k] += red[t][8 + k];
            }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            atomicAdd(sum + 8 * threadIdx.x + k, ts[k]);
            atomicAdd(sumsq + 8 * threadIdx.x + k, tq[k]);
        }
    }
}

// ----------------------------------------------------------------------------- forward apply
// Batch statistics -> mean and 1/std of a channel (fp64: the variance is E[y^2] - E[y]^2 of sums over up
// to 10^8 rows).  inv_n = 1/count is divided on the host (the same correctly rounded value; an fp64
// division on the device is a long chain of the GPU's slow fp64 operations), and 1/std is one fp64
// sequence instead of a root and a division.
__device__ __forceinline__ void finalize_channel(float sum, float sumsq, double inv_n, float eps, float& mean,
                                                 float& invstd)
{
    const double m = (double)sum * inv_n;
    double var = (double)sumsq * inv_n - m * m;
    if (var < 0.0) var = 0.0;
    mean = (float)m;
    invstd = (float)rsqrt(var + (double)eps);
}

__global__ void bn_fwd_finalize_kernel(double inv_n, int C, float eps, const float* __restrict__ sum,
                                       const float* __restrict__ sumsq, float* __restrict__ save_mean,
                                       float* __restrict__ save_invstd)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    finalize_channel(sum[c], sumsq[c], inv_n, eps, save_mean[c], save_invstd[c]);
}


// The same finalize from a convolution's per-CTA partials part[nparts][2][C]: the
// fixed-order partial sums (partials_colsum, rounded to fp32 as dbl_conv_fwd stores
// them), then mean and 1/std exactly as above.
__global__ void __launch_bounds__(dbl::dev::kPartialsThreads) bn_fwd_finalize_parts_kernel(double inv_n, int C, float eps,
                                                                    const float* __restrict__ part, int nparts,
                                                                    float* __restrict__ save_mean,
                                                                    float* __restrict__ save_invstd)
{
    float sum, sumsq;
    const int c = dbl::dev::partials_colsum(part, nparts, C, sum, sumsq);
    if (c < 0) return;
    finalize_channel(sum, sumsq, inv_n, eps, save_mean[c], save_invstd[c]);
}

// Thread t of a CTA owns channel group g = t % (C/8) (8 channels, one 16-byte
// vector) and visits rows t / (C/8), + rows-per-CTA-step, ...; a warp covers
// consecutive vectors of consecutive rows, so every access is coalesced, and the
// channel's scale and shift stay in registers.
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
    bn_apply_kernel(const act_t* __restrict__ y, const act_t* __restrict__ res,
                    act_t* __restrict__ out, int count, int C, int relu, int reverse, const float* __restrict__ gamma,
                    const float* __restrict__ beta, const float* __restrict__ mean, const float* __restrict__ invstd)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    extern __shared__ float4 chan4[];
    float* chan = reinterpret_cast<float*>(chan4);  // [scale, shift][C]
    for (int c = threadIdx.x; c < C; c += kThreads)
        bn_scale_shift(gamma[c], beta[c], mean[c], invstd[c], chan[c], chan[C + c]);
    __syncthreads();
    const int groups = C / 8;
    const int g = threadIdx.x % groups;
    const int rstep = kThreads / groups;
    float sc[8], sh[8];
    load8(chan + 8 * g, sc);
    load8(chan + C + 8 * g, sh);
    const int step = gridDim.x * rstep;
    auto emit = [&](const uint4& yv, const uint4& rv, int v) {
        float f[8], rr[8];
        unpack8(yv, f);
        unpack8(rv, rr);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float o = __fadd_rn(__fmaf_rn(f[k], sc[k], sh[k]), rr[k]);
            f[k] = (relu && !(o > 0.f)) ? 0.f : o;
        }
        reinterpret_cast<uint4*>(out)[v] = pack8(f);
    };
    const uint4 zero = make_uint4(0, 0, 0, 0);  // bf16 +0 in every lane
    int r = blockIdx.x * rstep + threadIdx.x / groups;
    const int base = reverse ? count - 1 : 0, dir = reverse ? -1 : 1;
    for (; r + (kUnroll - 1) * step < count; r += kUnroll * step) {
        uint4 yv[kUnroll], rv[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int v = (base + dir * (r + u * step)) * groups + g;
            yv[u] = __ldcs(reinterpret_cast<const uint4*>(y) + v);
            rv[u] = res ? __ldcs(reinterpret_cast<const uint4*>(res) + v) : zero;
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) emit(yv[u], rv[u], (base + dir * (r + u * step)) * groups + g);
    }
    for (; r < count; r += step) {
        const int v = (base + dir * r) * groups + g;
        emit(__ldcs(reinterpret_cast<const uint4*>(y) + v), res ? __ldcs(reinterpret_cast<const uint4*>(res) + v) : zero,
             v);
    }
}

// Finalize and apply in one launch, for small tensors whose convolution left few partials: every CTA takes 32
// channels (64 bytes of a row) and a run of the rows, and adds up its channels' partials for itself with the
// finalize's own tree (the same bits).  The partials come from L2 once per CTA, 256 bytes each, against a
// launch that reads them once.  576 rows of 512 channels, 32 partials: 5.2 -> 3.6 us.
constexpr int kFwdSliceC = 32, kFwdSliceRows = kThreads * 8 / kFwdSliceC;

__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
    bn_apply_parts_kernel(const act_t* __restrict__ y, const act_t* __restrict__ res, act_t* __restrict__ out,
                          int count, int C, int relu, double inv_n, float eps, const float* __restrict__ part,
                          int nparts, const float* __restrict__ gamma, const float* __restrict__ beta,
                          float* __restrict__ save_mean, float* __restrict__ save_invstd)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    __shared__ __align__(16) float chan[2][kFwdSliceC];  // scale, shift
    const int slices = C / kFwdSliceC, c0 = blockIdx.x % slices * kFwdSliceC;
    const int block = blockIdx.x / slices, blocks = gridDim.x / slices;
    float sum, sumsq;
    dbl::dev::partials_colsum32(part, nparts, C, c0, sum, sumsq);
    if (threadIdx.x < kFwdSliceC) {
        const int c = c0 + threadIdx.x;
        float m, is;
        finalize_channel(sum, sumsq, inv_n, eps, m, is);
        if (block == 0) {
            save_mean[c] = m;
            save_invstd[c] = is;
        }
        bn_scale_shift(gamma[c], beta[c], m, is, chan[0][threadIdx.x], chan[1][threadIdx.x]);
    }
    __syncthreads();
    const int vl = threadIdx.x % (kFwdSliceC / 8), groups = C / 8, g = c0 / 8 + vl;
    float sc[8], sh[8];
    load8(&chan[0][8 * vl], sc);
    load8(&chan[1][8 * vl], sh);
    const int step = blocks * kFwdSliceRows;
    constexpr int U = kUnroll;
    for (int r = block * kFwdSliceRows + threadIdx.x / (kFwdSliceC / 8); r < count; r += U * step) {
        uint4 yv[U], rv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t v = (int64_t)(r + u * step) * groups + g;
            const bool in = r + u * step < count;
            yv[u] = in ? __ldcs(reinterpret_cast<const uint4*>(y) + v) : make_uint4(0, 0, 0, 0);
            rv[u] = in && res ? __ldcs(reinterpret_cast<const uint4*>(res) + v) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (r + u * step < count) {
                float f[8], rr[8];
                unpack8(yv[u], f);
                unpack8(rv[u], rr);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float o = __fadd_rn(__fmaf_rn(f[k], sc[k], sh[k]), rr[k]);
                    f[k] = (relu && !(o > 0.f)) ? 0.f : o;
                }
                reinterpret_cast<uint4*>(out)[(int64_t)(r + u * step) * groups + g] = pack8(f);
            }
    }
}

// ----------------------------------------------------------------------------- backward
// Where the ReLU mask comes from: none (no ReLU), the stored output (out > 0),
// or, when there is no stored output (a BatchNorm without a residual), y,
// recomputed exactly as the forward pass decided it: y*scale + shift > 0 with
// the same fp32 operations.
enum MaskMode : int { kMaskNone = 0, kMaskOut = 1, kMaskY = 2 };

// The raw 16-byte vectors behind one 8-channel group of g = (dout [+ dout2]) * [out > 0]
// and of the BatchNorm input y; loaded together so that several rows' loads are in flight.
struct Vec8 {
    uint4 d, d2, o, y;
};

// One 16-byte vector.  KEEP: the apply pass reads the tensor again, so its lines stay in L2; otherwise
// they leave it first.
template <bool KEEP>
__device__ __forceinline__ uint4 load_vec(const act_t* p, int v)
{
    const uint4* q = reinterpret_cast<const uint4*>(p) + v;
    return KEEP ? __ldg(q) : __ldcs(q);
}

template <int MASK, bool KEEP_G, bool KEEP_Y>
__device__ __forceinline__ void load_g_raw(const act_t* dout, const act_t* dout2,
                                           const act_t* out, const act_t* y, int v, Vec8& g, Vec8& yv)
{
    g.d = load_vec<KEEP_G>(dout, v);
    g.d2 = dout2 ? load_vec<KEEP_G>(dout2, v) : make_uint4(0, 0, 0, 0);
    g.o = MASK == kMaskOut ? load_vec<KEEP_G>(out, v) : make_uint4(0, 0, 0, 0);
    yv.y = load_vec<KEEP_Y>(y, v);
}

template <int MASK>
struct ReluMask {
    float sc[MASK == kMaskY ? 8 : 1], sh[MASK == kMaskY ? 8 : 1];

    // s: [scale, shift][ld] in shared memory (stage_relu), c: the thread's first channel
    __device__ __forceinline__ void init(const float* s, int ld, int c)
    {
        if constexpr (MASK == kMaskY) {
            load8(s + c, sc);
            load8(s + ld + c, sh);
        }
    }
};

// Channels c0 .. c0 + n - 1 of the recomputed mask's scale and shift: s[0..n) and s[n..2n).
template <int MASK>
__device__ __forceinline__ void stage_relu(const float* gamma, const float* beta, const float* mean,
                                           const float* invstd, int c0, int n, float* s)
{
    if constexpr (MASK == kMaskY)
        for (int c = threadIdx.x; c < n; c += kThreads)
            bn_scale_shift(gamma[c0 + c], beta[c0 + c], mean[c0 + c], invstd[c0 + c], s[c], s[n + c]);
}

template <int MASK>
__device__ __forceinline__ void combine_g(const Vec8& raw, const float (&y)[8], bool two, const ReluMask<MASK>& m,
                                          float (&g)[8])
{
    unpack8(raw.d, g);
    if (two) {
        float h[8];
        unpack8(raw.d2, h);
#pragma unroll
        for (int k = 0; k < 8; ++k) g[k] += h[k];
    }
    if constexpr (MASK == kMaskY) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (!(__fmaf_rn(y[k], m.sc[k], m.sh[k]) > 0.f)) g[k] = 0.f;
    } else if constexpr (MASK == kMaskOut) {
        float o[8];
        unpack8(raw.o, o);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (!(o[k] > 0.f)) g[k] = 0.f;
    }
}

// sg += g, sgc += g*(y - mean)  (the 1/std factor is applied once per partial)
// WRITE_G: also store g (bf16) at vector v of g_out.  The sums are of the fp32 g (the
// dgamma, dbeta outputs keep fp32 accuracy); the apply pass then reads the stored g.
template <int MASK, bool WRITE_G>
__device__ __forceinline__ void accumulate_g(const Vec8& graw, const Vec8& yraw, bool two, const ReluMask<MASK>& relu,
                                             const float (&mu)[8], float (&sg)[8], float (&sgc)[8],
                                             act_t* g_out, int v)
{
    float gg[8], yy[8];
    unpack8(yraw.y, yy);
    combine_g(graw, yy, two, relu, gg);
    if constexpr (WRITE_G) reinterpret_cast<uint4*>(g_out)[v] = pack8(gg);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        sg[k] += gg[k];
        sgc[k] = fmaf(gg[k], yy[k] - mu[k], sgc[k]);
    }
}

// Partial blk reduces the row chunks blk, blk + nblk, blk + 2*nblk, ... (a chunk
// is the kThreads/(C/8) rows one CTA covers in one step) into partial[blk][0..C)
// (sum g) and partial[blk][C..2C) (sum g*xhat); CTA b computes partials b,
// b + gridDim.x, ....  Interleaved chunks keep all CTAs streaming through the same
// region of the tensors, and each partial adds its rows in a fixed order, so the
// result does not depend on the grid.
// The rows are visited last to first: the data gradient before this pass wrote dout from
// row 0 on, so its end is still in L2, and the apply pass after it, which goes from row 0
// on, finds the rows visited last here.  What the apply pass reads again (y, and g or
// dout) is loaded and stored with the default cache policy, the rest evict-first.  Both
// passes at HBM rate before and after: a residual block's backward at 128 channels, batch 185,
// 28 x 28 (37 MB tensors) 320 -> 306 us, at 64 channels, batch 512, 56 x 56 (206 MB) 883 -> 865 us.
template <int MASK, bool WRITE_G>
__global__ void __launch_bounds__(kThreads, kReduceBlocksPerSM)
    bn_bwd_reduce_kernel(const act_t* __restrict__ dout, const act_t* __restrict__ dout2,
                         const act_t* __restrict__ out, const act_t* __restrict__ y, int count,
                         int C, const float* __restrict__ gamma, const float* __restrict__ beta,
                         const float* __restrict__ mean, const float* __restrict__ invstd, int nblk,
                         float* __restrict__ partial, act_t* __restrict__ g_out)
{
    extern __shared__ float4 chan4[];
    float* chan = reinterpret_cast<float*>(chan4);  // [mean (, scale, shift)][C]
    for (int c = threadIdx.x; c < C; c += kThreads) chan[c] = mean[c];
    stage_relu<MASK>(gamma, beta, mean, invstd, 0, C, chan + C);
    __syncthreads();
    const int groups = C / 8;
    const int g = threadIdx.x % groups;
    const int rstep = kThreads / groups;
    ReluMask<MASK> rm;
    rm.init(chan + C, C, 8 * g);
    float mu[8];
    load8(chan + 8 * g, mu);
    __shared__ float red[kThreads][17];
    const int cstep = nblk * rstep;  // rows from one chunk of a partial to its next
    constexpr int U = kReduceUnroll;  // chunks whose loads are in flight together
    for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    float sg[8] = {}, sgx[8] = {};
    int r = blk * rstep + threadIdx.x / groups;
    const int last = count - 1;
    for (; r + (U - 1) * cstep < count; r += U * cstep) {
        Vec8 gg[U], yy[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            load_g_raw<MASK, !WRITE_G, true>(dout, dout2, out, y, (last - (r + u * cstep)) * groups + g, gg[u], yy[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
            accumulate_g<MASK, WRITE_G>(gg[u], yy[u], dout2 != nullptr, rm, mu, sg, sgx, g_out,
                                        (last - (r + u * cstep)) * groups + g);
    }
    for (; r < count; r += cstep) {
        Vec8 gg, yy;
        load_g_raw<MASK, !WRITE_G, true>(dout, dout2, out, y, (last - r) * groups + g, gg, yy);
        accumulate_g<MASK, WRITE_G>(gg, yy, dout2 != nullptr, rm, mu, sg, sgx, g_out, (last - r) * groups + g);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        red[threadIdx.x][k] = sg[k];
        red[threadIdx.x][8 + k] = sgx[k];
    }
    __syncthreads();
    float* p = partial + (int64_t)blk * 2 * C;
    for (int i = threadIdx.x; i < 2 * C; i += kThreads) {  // one sum per thread, rows in order
        const int x = i >= C, c = i - x * C;
        float t = 0.f;
        for (int j = c / 8; j < rstep * groups; j += groups) t += red[j][8 * x + c % 8];
        p[i] = x ? t * invstd[c] : t;  // sum g*(y-mean) -> sum g*xhat
    }
    __syncthreads();
    }
}

// Max-pool backward and the reduce pass of the BatchNorm + ReLU before the pool, in one: a step takes
// 2x2 blocks of pixels (i, j) in place of rows, gathers their gradient from the windows (i..i+1, j..j+1)
// (maxpool_bwd_kernel's taps and order), stores it as da for the apply pass, and sums the stored values
// masked by y: at most kPoolParts partials, each over blocks in a fixed order, last to first.  Against
// its own memory traffic (two tensors of the pool's input and a half) at 0.85 of the copy bandwidth; the
// gather's instructions fill the rest.  Pool pass, reduce, finalize and apply with two gradients -> with this
// (us): 112x112x64, batch 512 917 -> 740 (with 256 partials in CTAs of 256 threads, two on some SMs, 853;
// one channel per operation 781; walking runs of rows, the lower windows kept and the next row copied ahead
// with cp.async, 798), batch 64 125 -> 104; 80x80, batch 512 472 -> 384; 144x144, batch 185 551 -> 447;
// 64x64, batch 64 44.7 -> 39.1, batch 16 19.2 -> 17.3.
constexpr int kPoolThreads = 512;
constexpr int64_t kPoolParts = 152;  // one CTA per SM
__global__ void __launch_bounds__(kPoolThreads, 1)
    bn_pool_bwd_reduce_kernel(const act_t* __restrict__ dp, const act_t* __restrict__ dp2,
                              const uint8_t* __restrict__ arg, const act_t* __restrict__ y, int n, int H, int W,
                              int C, const float* __restrict__ gamma, const float* __restrict__ beta,
                              const float* __restrict__ mean, const float* __restrict__ invstd, int nblk,
                              float* __restrict__ partial, act_t* __restrict__ da)
{
    extern __shared__ float4 chan4[];
    float* chan = reinterpret_cast<float*>(chan4);  // [mean, scale, shift][C]
    for (int c = threadIdx.x; c < C; c += kPoolThreads) chan[c] = mean[c];
    stage_relu<kMaskY>(gamma, beta, mean, invstd, 0, C, chan + C);
    __syncthreads();
    const int groups = C / 8;
    const int g = threadIdx.x % groups;
    const int rstep = kPoolThreads / groups;
    ReluMask<kMaskY> rm;
    rm.init(chan + C, C, 8 * g);
    float mu[8];
    load8(chan + 8 * g, mu);
    float2 sc2[4], sh2[4], mu2[4];  // two channels per operation
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        sc2[k] = make_float2(rm.sc[2 * k], rm.sc[2 * k + 1]);
        sh2[k] = make_float2(rm.sh[2 * k], rm.sh[2 * k + 1]);
        mu2[k] = make_float2(-mu[2 * k], -mu[2 * k + 1]);
    }
    __shared__ float red[kPoolThreads][17];
    const int P = (H + 1) / 2, Q = (W + 1) / 2;
    const int total = n * P * Q, cstep = nblk * rstep;
    const int step_j = cstep % Q, step_i = cstep / Q % P, step_b = cstep / Q / P;
    const int win_row = Q * groups, px_row = W * groups;
    for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        float2 sg[4] = {}, sgx[4] = {};
        int r = blk * rstep + threadIdx.x / groups;
        const int first = max(total - 1 - r, 0);
        int j = first % Q, i = first / Q % P, b = first / Q / P;
        for (; r < total; r += cstep) {
            const bool r1 = i + 1 < P, c1 = j + 1 < Q;              // windows below and to the right
            const bool h1 = 2 * i + 1 < H, w1 = 2 * j + 1 < W;      // pixels
            const int o = ((b * P + i) * Q + j) * groups + g;       // window (i, j)
            const int v = ((b * H + 2 * i) * W + 2 * j) * groups + g;  // pixel (2i, 2j)
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            uint4 gv[4], gv2[4], yv[4];
            uint2 av[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const bool ok = (t < 2 || r1) && (t % 2 == 0 || c1);
                const int ot = o + (t >> 1) * win_row + (t & 1) * groups;
                gv[t] = ok ? __ldg(reinterpret_cast<const uint4*>(dp) + ot) : zero;
                gv2[t] = ok && dp2 ? __ldg(reinterpret_cast<const uint4*>(dp2) + ot) : zero;
                av[t] = ok ? __ldg(reinterpret_cast<const uint2*>(arg) + ot) : make_uint2(~0u, ~0u);
                yv[t] = (t < 2 || h1) && (t % 2 == 0 || w1)
                            ? __ldg(reinterpret_cast<const uint4*>(y) + v + (t >> 1) * px_row + (t & 1) * groups)
                            : zero;
            }
            // window t's gradient: dp [+ dp2]
            auto window = [&](int t, float (&f)[8]) {
                unpack8(gv[t], f);
                if (dp2) {
                    float f2[8];
                    unpack8(gv2[t], f2);
#pragma unroll
                    for (int k = 0; k < 8; k += 2) {
                        const float2 t2 = dbl::dev::add2(make_float2(f[k], f[k + 1]), make_float2(f2[k], f2[k + 1]));
                        f[k] = t2.x, f[k + 1] = t2.y;
                    }
                }
            };
            auto pixel = [&](int t, const float (&acc)[8]) {
                const uint4 packed = pack8(acc);
                reinterpret_cast<uint4*>(da)[v + (t >> 1) * px_row + (t & 1) * groups] = packed;
                float gg[8], yy[8];
                unpack8(packed, gg);
                unpack8(yv[t], yy);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 y2 = make_float2(yy[2 * k], yy[2 * k + 1]);
                    const float2 pre = dbl::dev::fma2(y2, sc2[k], sh2[k]);
                    const float2 g2 = make_float2(pre.x > 0.f ? gg[2 * k] : 0.f, pre.y > 0.f ? gg[2 * k + 1] : 0.f);
                    sg[k] = dbl::dev::add2(sg[k], g2);
                    sgx[k] = dbl::dev::fma2(g2, dbl::dev::add2(y2, mu2[k]), sgx[k]);
                }
            };
            float f[8], acc01[8] = {}, acc10[8] = {}, acc11[8] = {};
            window(0, f);
            {
                float acc00[8] = {};
                dbl::dev::add_if_tap(acc00, f, av[0], 4);
                pixel(0, acc00);
            }
            dbl::dev::add_if_tap(acc01, f, av[0], 5);
            dbl::dev::add_if_tap(acc10, f, av[0], 7);
            dbl::dev::add_if_tap(acc11, f, av[0], 8);
            window(1, f);
            dbl::dev::add_if_tap(acc01, f, av[1], 3);
            dbl::dev::add_if_tap(acc11, f, av[1], 6);
            if (w1) pixel(1, acc01);
            window(2, f);
            dbl::dev::add_if_tap(acc10, f, av[2], 1);
            dbl::dev::add_if_tap(acc11, f, av[2], 2);
            if (h1) pixel(2, acc10);
            window(3, f);
            dbl::dev::add_if_tap(acc11, f, av[3], 0);
            if (h1 && w1) pixel(3, acc11);
            // cstep blocks back
            j -= step_j;
            i -= step_i;
            b -= step_b;
            if (j < 0) j += Q, --i;
            if (i < 0) i += P, --b;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            red[threadIdx.x][2 * k] = sg[k].x;
            red[threadIdx.x][2 * k + 1] = sg[k].y;
            red[threadIdx.x][8 + 2 * k] = sgx[k].x;
            red[threadIdx.x][8 + 2 * k + 1] = sgx[k].y;
        }
        __syncthreads();
        float* p = partial + (int64_t)blk * 2 * C;
        for (int e = threadIdx.x; e < 2 * C; e += kPoolThreads) {  // one sum per thread, of four of every fourth row
            const int x = e >= C, c = e - x * C;
            float t[4] = {};
            for (int q = 0; q < rstep; q += 4)  // rstep: a power of two, 4 or more (at most 1024 channels)
#pragma unroll
                for (int k = 0; k < 4; ++k) t[k] += red[(q + k) * groups + c / 8][8 * x + c % 8];
            const float u = (t[0] + t[1]) + (t[2] + t[3]);
            p[e] = x ? u * invstd[c] : u;
        }
        __syncthreads();
    }
}

// dy = k1*(g - sum(g)/n - xhat*sum(g*xhat)/n), xhat = (y - mean)*invstd, as A*g + B*y + C;
// inv_n = 1/count, divided on the host.
__device__ __forceinline__ void bwd_coefficients(double sg, double sgx, double inv_n, float gamma, float invstd,
                                                 float mean, float& a, float& b, float& c)
{
    const double k1 = (double)gamma * (double)invstd;
    const double kb = -k1 * (double)invstd * (sgx * inv_n);
    a = (float)k1;
    b = (float)kb;
    c = (float)(-k1 * (sg * inv_n) - kb * (double)mean);
}

// Fixed-order sum of the partials [nblk][2][C] (partials_colsum), then dgamma,
// dbeta and the three per-channel coefficients (A, B, C) of the apply pass
// dy = A*g + B*y + C.
__global__ void __launch_bounds__(dbl::dev::kPartialsThreads) bn_bwd_finalize_kernel(
    const float* __restrict__ partial, int nblk, int C, double inv_n, const float* __restrict__ gamma,
    const float* __restrict__ mean, const float* __restrict__ invstd, float* __restrict__ dgamma,
    float* __restrict__ dbeta, float* __restrict__ coef)
{
    double sg, sgx;
    const int c = dbl::dev::partials_colsum(partial, nblk, C, sg, sgx);
    if (c < 0) return;
    dbeta[c] = (float)sg;
    dgamma[c] = (float)sgx;
    bwd_coefficients(sg, sgx, inv_n, gamma[c], invstd[c], mean[c], coef[c], coef[C + c], coef[2 * C + c]);
}

template <int MASK>
__global__ void __launch_bounds__(kThreads, kBwdBlocksPerSM)
    bn_bwd_apply_kernel(const act_t* __restrict__ dout, const act_t* __restrict__ dout2,
                        const act_t* __restrict__ out, const act_t* __restrict__ y, int count,
                        int C, const float* __restrict__ gamma, const float* __restrict__ beta,
                        const float* __restrict__ mean, const float* __restrict__ invstd,
                        const float* __restrict__ coef, act_t* __restrict__ dy, act_t* __restrict__ dres)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    extern __shared__ float4 chan4[];
    float* chan = reinterpret_cast<float*>(chan4);  // [A, B, C (, scale, shift)][C]
    for (int c = threadIdx.x; c < 3 * C; c += kThreads) chan[c] = coef[c];
    stage_relu<MASK>(gamma, beta, mean, invstd, 0, C, chan + 3 * C);
    __syncthreads();
    const int groups = C / 8;
    const int g = threadIdx.x % groups;
    const int rstep = kThreads / groups;
    ReluMask<MASK> rm;
    rm.init(chan + 3 * C, C, 8 * g);
    float ca[8], cb[8], cc[8];
    load8(chan + 8 * g, ca);
    load8(chan + C + 8 * g, cb);
    load8(chan + 2 * C + 8 * g, cc);
    const int step = gridDim.x * rstep;
    auto emit = [&](const Vec8& graw, const Vec8& yraw, int v) {
        float gg[8], yy[8], d[8];
        unpack8(yraw.y, yy);
        combine_g(graw, yy, dout2 != nullptr, rm, gg);
#pragma unroll
        for (int k = 0; k < 8; ++k) d[k] = fmaf(ca[k], gg[k], fmaf(cb[k], yy[k], cc[k]));
        reinterpret_cast<uint4*>(dy)[v] = pack8(d);
        if (dres) __stcs(reinterpret_cast<uint4*>(dres) + v, pack8(gg));
    };
    int r = blockIdx.x * rstep + threadIdx.x / groups;
    for (; r + (kUnroll - 1) * step < count; r += kUnroll * step) {
        Vec8 gg[kUnroll], yy[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) load_g_raw<MASK, false, false>(dout, dout2, out, y, (r + u * step) * groups + g, gg[u], yy[u]);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) emit(gg[u], yy[u], (r + u * step) * groups + g);
    }
    for (; r < count; r += step) {
        Vec8 gg, yy;
        load_g_raw<MASK, false, false>(dout, dout2, out, y, r * groups + g, gg, yy);
        emit(gg, yy, r * groups + g);
    }
}

// ----------------------------------------------------------------------------- small tensors
// Backward of small tensors in one launch instead of three: a cluster of CL CTAs owns 32 channels, each
// CTA an equal run of the rows.  Both passes over the rows read global memory (the second finds its
// CTA's rows in L1 and L2); between them the CTAs add up their channel sums through distributed shared
// memory, in rank order, and each forms the three coefficients of the apply pass for itself.  Bound
// by latency: three launches of the general path cost about 3 us each before they move a byte.
// General path -> here, bwd without / with a second gradient and g stored (us): 576 rows of 512 channels
// 11.1 -> 5.4 / 10.8 -> 5.8; 4608 of 512 13.2 -> 9.8 / 12.8 -> 11.2 (stays); 4608 of 256 11.4 -> 7.8 /
// 11.1 -> 8.8; 12,800 of 256 13.6 -> 12.5 / 13.5 -> 14.0 (stays); 16,384 of 128 11.2 -> 11.6 (stays).
constexpr int kSliceC = 32;                    // channels of a slice: 64 bytes of a row
constexpr int kSliceVec = kSliceC / 8;         // 16-byte vectors of a slice row
constexpr int kSliceRows = kThreads / kSliceVec;  // rows a CTA covers in one step

template <int MASK, bool WRITE_G>
__global__ void __launch_bounds__(kThreads, 2)
    bn_bwd_cluster_kernel(const act_t* __restrict__ dout, const act_t* __restrict__ dout2,
                          const act_t* __restrict__ out, const act_t* __restrict__ y, int count, int C,
                          double inv_n, const float* __restrict__ gamma, const float* __restrict__ beta,
                          const float* __restrict__ mean, const float* __restrict__ invstd,
                          float* __restrict__ dgamma, float* __restrict__ dbeta, act_t* __restrict__ dy,
                          act_t* dres, int CL)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    __shared__ float red[kThreads / 32][2][kSliceC];
    __shared__ float tot[2][kSliceC];   // this CTA's sums, read by the whole cluster
    __shared__ double all[2][kSliceC];  // the cluster's
    __shared__ __align__(16) float coef[3][kSliceC];
    const int rank = (int)dbl::dev::cluster_ctarank(), slice = blockIdx.x / CL;
    const int c0 = slice * kSliceC, vl = threadIdx.x % kSliceVec, g = c0 / 8 + vl, groups = C / 8;
    const int per = (count + CL - 1) / CL, r0 = rank * per, r1 = min(count, r0 + per);
    const bool two = dout2 != nullptr;
    __shared__ __align__(16) float chan[3 * kSliceC];  // mean (, scale, shift)
    if (threadIdx.x < kSliceC) chan[threadIdx.x] = mean[c0 + threadIdx.x];
    stage_relu<MASK>(gamma, beta, mean, invstd, c0, kSliceC, chan + kSliceC);
    __syncthreads();
    ReluMask<MASK> rm;
    rm.init(chan + kSliceC, kSliceC, 8 * vl);
    float mu[8];
    load8(chan + 8 * vl, mu);
    constexpr int U = 4;  // rows whose loads are in flight together
    float sg[8] = {}, sgx[8] = {};
    for (int r = r0 + threadIdx.x / kSliceVec; r < r1; r += U * kSliceRows) {
        Vec8 gg[U], yy[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (r + u * kSliceRows < r1)
                load_g_raw<MASK, true, true>(dout, dout2, out, y, (r + u * kSliceRows) * groups + g, gg[u], yy[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (r + u * kSliceRows < r1)
                accumulate_g<MASK, WRITE_G>(gg[u], yy[u], two, rm, mu, sg, sgx, dres,
                                            (r + u * kSliceRows) * groups + g);
    }
    // lanes that share a vector, then the warps in order
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int o = kSliceVec; o < 32; o <<= 1) {
            sg[k] += __shfl_xor_sync(0xffffffffu, sg[k], o);
            sgx[k] += __shfl_xor_sync(0xffffffffu, sgx[k], o);
        }
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (lane < kSliceVec)
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            red[warp][0][8 * vl + k] = sg[k];
            red[warp][1][8 * vl + k] = sgx[k];
        }
    __syncthreads();
    if (threadIdx.x < 2 * kSliceC) {
        const int st = threadIdx.x / kSliceC, c = threadIdx.x % kSliceC;
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) t += red[w][st][c];
        tot[st][c] = st ? t * invstd[c0 + c] : t;  // sum g*(y-mean) -> sum g*xhat
    }
    __syncwarp();
    dbl::dev::cluster_sync_all();
    if (threadIdx.x < 2 * kSliceC) {  // one sum per thread
        const int st = threadIdx.x / kSliceC, c = threadIdx.x % kSliceC;
        float v[16];
#pragma unroll
        for (int r = 0; r < 16; ++r)
            v[r] = r < CL ? dbl::dev::ld_cluster_f32(dbl::dev::mapa_shared(dbl::dev::smem_u32(&tot[st][c]), r)) : 0.f;
        dbl::dev::Sum3 t{0.f, 0.f, 0.f};
#pragma unroll
        for (int r = 0; r < 16; ++r)
            if (r < CL) t = dbl::dev::sum_add(t, v[r]);
        double sum = dbl::dev::sum_f64(t);
        if (!dbl::dev::sum_held(t)) {  // beyond fp32's range, or not a number
            sum = 0.0;
#pragma unroll
            for (int r = 0; r < 16; ++r)
                if (r < CL) sum += (double)v[r];
        }
        all[st][c] = sum;
    }
    __syncthreads();
    if (threadIdx.x < kSliceC) {
        const int c = threadIdx.x;
        const double sums[2] = {all[0][c], all[1][c]};
        if (rank == 0) {
            dbeta[c0 + c] = (float)sums[0];
            dgamma[c0 + c] = (float)sums[1];
        }
        bwd_coefficients(sums[0], sums[1], inv_n, gamma[c0 + c], invstd[c0 + c], mean[c0 + c], coef[0][c], coef[1][c],
                         coef[2][c]);
    }
    __syncthreads();
    float ca[8], cb[8], cc[8];
    load8(&coef[0][8 * vl], ca);
    load8(&coef[1][8 * vl], cb);
    load8(&coef[2][8 * vl], cc);
    for (int r = r0 + threadIdx.x / kSliceVec; r < r1; r += 2 * kSliceRows) {
        Vec8 gg[2], yy[2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (r + u * kSliceRows < r1) {
                const int v = (r + u * kSliceRows) * groups + g;
                if constexpr (WRITE_G) {  // the g this thread stored, as the general path reads it back
                    gg[u].d = __ldcg(reinterpret_cast<const uint4*>(dres) + v);
                    yy[u].y = load_vec<true>(y, v);
                } else {
                    load_g_raw<MASK, true, true>(dout, dout2, out, y, v, gg[u], yy[u]);
                }
            }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (r + u * kSliceRows < r1) {
                float f[8], x[8], d[8];
                unpack8(yy[u].y, x);
                if constexpr (WRITE_G)
                    unpack8(gg[u].d, f);
                else
                    combine_g(gg[u], x, two, rm, f);
#pragma unroll
                for (int k = 0; k < 8; ++k) d[k] = fmaf(ca[k], f[k], fmaf(cb[k], x[k], cc[k]));
                reinterpret_cast<uint4*>(dy)[(r + u * kSliceRows) * groups + g] = pack8(d);
            }
    }
    dbl::dev::cluster_sync_all();  // no CTA leaves while another may still read its sums
}

// CTAs per cluster of the one-launch backward, or 0 for the general path: the channels must come in
// whole slices, and a CTA's rows (kClusterRows, with g to store kClusterRowsG) stay few enough that its
// two passes cost less than the two launches saved.  (A device that cannot place the cluster takes the general
// path.)
constexpr int kClusterRows = 800, kClusterRowsG = 512;

int bwd_cluster(int64_t count, int C, bool with_g)
{
    if (C % kSliceC) return 0;
    const int cl = C >= 512 ? 8 : 16;  // at least 64 CTAs; sixteen is above the portable cluster size
    return count <= (int64_t)cl * (with_g ? kClusterRowsG : kClusterRows) ? cl : 0;
}

int bn_grid(int64_t nvec, int per_sm = kBlocksPerSM)
{
    int64_t b = (nvec + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)dbl::sm_count() * per_sm;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

// One wave of CTAs that take the same number of partials each (more partials than
// resident CTAs would leave some of them a second round alone).
int reduce_grid(int64_t nblk)
{
    const int64_t cap = (int64_t)dbl::sm_count() * kReduceBlocksPerSM;
    const int64_t per_cta = (nblk + cap - 1) / cap;
    return (int)((nblk + per_cta - 1) / per_cta);
}

// Forward in one launch (bn_apply_parts_kernel)?  Whole rows stream better than 64-byte slices, and above ~100
// partials every CTA's own sum costs what the second launch does (us, two launches -> one): 2 MB with 32 /
// 100 / 152 partials 5.9 -> 4.4, 6.1 -> 5.2, 6.1 -> 6.0; 6.6 MB 6.6 -> 5.6, 6.8 -> 6.4, 6.9 -> 7.1; 12.8 MB with 32
// 7.8 -> 7.0, with 152 8.0 -> 8.5.  The line lies where one launch is still the better one with most partials.
bool fwd_one_launch(int64_t count, int C, int nparts)
{
    return C % kFwdSliceC == 0 && nparts <= 104 && count * C * (int64_t)sizeof(act_t) <= (int64_t)8 << 20;
}

int apply_reversed(const dbl_bn_shape* s) { return s->count * s->c * (int64_t)sizeof(act_t) > kReverseAboveBytes; }

int check_shape(const dbl_bn_shape* s, const char* who)
{
    if (!s || s->count < 0 || s->c <= 0) return dbl::set_error(DBL_ERR_INVALID, "%s: bad shape", who);
    if (s->c % 8 != 0 || s->c > kMaxC || (kThreads % (s->c / 8)) != 0)
        return dbl::set_error(DBL_ERR_UNSUPPORTED, "%s: channel count %d (need a multiple of 8 dividing 2048)", who,
                              s->c);
    // the streaming kernels index 16-byte vectors (and rows, plus one grid step, or the
    // reduce's kReduceUnroll chunk strides of at most 512 partials) in 32 bits
    if (s->count * (s->c / 8) + (int64_t)kThreads * dbl::sm_count() * kBlocksPerSM * kUnroll +
            (int64_t)kThreads * 512 * kReduceUnroll >=
        ((int64_t)1 << 31))
        return dbl::set_error(DBL_ERR_UNSUPPORTED, "%s: %lld x %d elements exceed the 2^31-vector limit", who,
                              (long long)s->count, s->c);
    return DBL_OK;
}

// Backward reduce split: a fixed function of the shape (so the workspace size
// and the summation order do not depend on the device): one partial per 2048
// 8-channel vectors (8 per thread), at most kMaxBwdParts.  The cap is below the
// reduce's resident CTAs on this GPU (two per SM), so a large tensor gets one
// partial per CTA; a cap of 512 gave those CTAs two partials each and the
// finalize twice the partials to add (8 us per call at layer4, batch 512).
constexpr int64_t kMaxBwdParts = 256;
int64_t bwd_blocks(int64_t count, int C)
{
    if (count <= 0 || C <= 0) return 1;
    const int64_t b = (count * (C / 8) + 2047) / 2048;
    return b < 1 ? 1 : b > kMaxBwdParts ? kMaxBwdParts : b;
}

// The passes after the reduce: fixed-order finalize and apply.
template <int MASK>
int bwd_finish(const dbl_bn_shape* s, const void* dout, const void* dout2, const void* y, const void* out,
               const float* gamma, const float* beta, const float* mean, const float* invstd, void* dy, float* dgamma,
               float* dbeta, float* partial, float* coef, int64_t nblk, cudaStream_t st)
{
    using namespace dbl;
    const int C = s->c;
    auto bd = [](const void* p) { return static_cast<const act_t*>(p); };
    bn_bwd_finalize_kernel<<<(C + dbl::dev::kPartialsChannels - 1) / dbl::dev::kPartialsChannels,
                             dbl::dev::kPartialsThreads, 0, st>>>(partial, (int)nblk, C, 1.0 / (double)s->count, gamma,
                                                                  mean, invstd, dgamma, dbeta, coef);
    if (int rc = launch_check("bn_bwd_finalize launch")) return rc;
    bn_bwd_apply_kernel<MASK><<<bn_grid(s->count * C / 8, kBwdBlocksPerSM), kThreads,
                                (MASK == kMaskY ? 5 : 3) * C * sizeof(float), st>>>(
        bd(dout), bd(dout2), bd(out), bd(y), (int)s->count, C, gamma, beta, mean, invstd, coef,
        static_cast<act_t*>(dy), nullptr);
    return launch_check("bn_bwd_apply launch");
}

template <int MASK>
int bwd_launch_mask(const dbl_bn_shape* s, const void* dout, const void* dout2, const void* y, const void* out,
                    const float* gamma, const float* beta, const float* mean, const float* invstd, void* dy,
                    void* dresidual, float* dgamma, float* dbeta, float* partial, float* coef, int64_t nblk,
                    cudaStream_t st)
{
    using namespace dbl;
    const int C = s->c;
    auto bd = [](const void* p) { return static_cast<const act_t*>(p); };
    // When the caller wants g (the residual branch's gradient), the reduce pass stores it and the
    // apply pass reads it back instead of re-reading dout, dout2 and out.
    act_t* g_store = static_cast<act_t*>(dresidual);
    const int cl = bwd_cluster(s->count, C, g_store != nullptr);
    if (cl && (g_store ? cluster_held<bn_bwd_cluster_kernel<MASK, true>>(cl, kThreads, 0)
                       : cluster_held<bn_bwd_cluster_kernel<MASK, false>>(cl, kThreads, 0))) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cl;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C / kSliceC * cl);
        cfg.blockDim = dim3(kThreads);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        auto k = g_store ? bn_bwd_cluster_kernel<MASK, true> : bn_bwd_cluster_kernel<MASK, false>;
        cudaError_t e = cl > 8 ? cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : cudaSuccess;
        if (e == cudaSuccess)
            e = cudaLaunchKernelEx(&cfg, k, bd(dout), bd(dout2), bd(out), bd(y), (int)s->count, C,
                                   1.0 / (double)s->count, gamma, beta, mean, invstd, dgamma, dbeta,
                                   static_cast<act_t*>(dy), g_store, cl);
        if (e != cudaSuccess) {
            count_launch();
            return cuda_check(e, "bn_bwd_cluster launch");
        }
        return launch_check("bn_bwd_cluster launch");
    }
    const size_t smem_r = (MASK == kMaskY ? 3 : 1) * C * sizeof(float);
    if (g_store)
        bn_bwd_reduce_kernel<MASK, true><<<reduce_grid(nblk), kThreads, smem_r, st>>>(
            bd(dout), bd(dout2), bd(out), bd(y), (int)s->count, C, gamma, beta, mean, invstd, (int)nblk, partial,
            g_store);
    else
        bn_bwd_reduce_kernel<MASK, false><<<reduce_grid(nblk), kThreads, smem_r, st>>>(
            bd(dout), bd(dout2), bd(out), bd(y), (int)s->count, C, gamma, beta, mean, invstd, (int)nblk, partial,
            nullptr);
    if (int rc = launch_check("bn_bwd_reduce launch")) return rc;
    if (g_store)
        return bwd_finish<kMaskNone>(s, g_store, nullptr, y, nullptr, gamma, beta, mean, invstd, dy, dgamma, dbeta,
                                     partial, coef, nblk, st);
    return bwd_finish<MASK>(s, dout, dout2, y, out, gamma, beta, mean, invstd, dy, dgamma, dbeta, partial, coef, nblk,
                            st);
}

// The three passes of the backward pass (reduce, fixed-order finalize, apply),
// with the ReLU mask taken from out, recomputed from y (out == NULL), or none.
int bwd_launch(const dbl_bn_shape* s, const void* dout, const void* dout2, const void* y, const void* out,
               const float* gamma, const float* beta, const float* mean, const float* invstd, void* dy, void* dresidual,
               float* dgamma, float* dbeta, float* partial, float* coef, int64_t nblk, cudaStream_t st)
{
    if (!s->relu)
        return bwd_launch_mask<kMaskNone>(s, dout, dout2, y, out, gamma, beta, mean, invstd, dy, dresidual, dgamma,
                                          dbeta, partial, coef, nblk, st);
    if (out)
        return bwd_launch_mask<kMaskOut>(s, dout, dout2, y, out, gamma, beta, mean, invstd, dy, dresidual, dgamma,
                                         dbeta, partial, coef, nblk, st);
    return bwd_launch_mask<kMaskY>(s, dout, dout2, y, out, gamma, beta, mean, invstd, dy, dresidual, dgamma, dbeta,
                                   partial, coef, nblk, st);
}

}  // namespace

namespace dbl {

int bn_fwd_finalize(int64_t count, int C, float eps, const float* sum, const float* sumsq, float* save_mean,
                    float* save_invstd, cudaStream_t st)
{
    bn_fwd_finalize_kernel<<<(C + 127) / 128, 128, 0, st>>>(1.0 / (double)count, C, eps, sum, sumsq, save_mean,
                                                            save_invstd);
    return launch_check("bn_fwd_finalize launch");
}

}  // namespace dbl

extern "C" {

int dbl_bn_stats(const dbl_bn_shape* s, const void* y, float* ch_sum, float* ch_sumsq, void* stream)
{
    using namespace dbl;
    int rc = check_shape(s, "bn_stats");
    if (rc) return rc;
    if (!y || !ch_sum || !ch_sumsq || !aligned16(y)) return set_error(DBL_ERR_INVALID, "bn_stats: bad pointer");
    cudaStream_t st = as_stream(stream);
    if ((rc = cuda_check(cudaMemsetAsync(ch_sum, 0, sizeof(float) * s->c, st), "bn_stats memset"))) return rc;
    if ((rc = cuda_check(cudaMemsetAsync(ch_sumsq, 0, sizeof(float) * s->c, st), "bn_stats memset"))) return rc;
    if (s->count == 0) return DBL_OK;
    bn_stats_kernel<<<bn_grid(s->count * s->c / 8), kThreads, 0, st>>>(static_cast<const act_t*>(y), s->count,
                                                                       s->c, ch_sum, ch_sumsq);
    return launch_check("bn_stats launch");
}

int dbl_bn_relu_fused(const dbl_bn_shape* s, const void* y, const float* ch_sum, const float* ch_sumsq,
                      const float* gamma, const float* beta, const void* residual, void* out, float* save_mean,
                      float* save_invstd, void* stream)
{
    using namespace dbl;
    int rc = check_shape(s, "bn_relu_fused");
    if (rc) return rc;
    if (!y || !out || !ch_sum || !ch_sumsq || !gamma || !beta || !save_mean || !save_invstd)
        return set_error(DBL_ERR_INVALID, "bn_relu_fused: null pointer");
    if (!aligned16(y) || !aligned16(out) || (residual && !aligned16(residual)))
        return set_error(DBL_ERR_INVALID, "bn_relu_fused: tensors must be 16-byte aligned");
    if (s->count == 0) return set_error(DBL_ERR_INVALID, "bn_relu_fused: empty batch has no statistics");
    cudaStream_t st = as_stream(stream);
    if ((rc = bn_fwd_finalize(s->count, s->c, s->eps, ch_sum, ch_sumsq, save_mean, save_invstd, st))) return rc;
    bn_apply_kernel<<<bn_grid(s->count * s->c / 8), kThreads, 2 * s->c * sizeof(float), st>>>(
        static_cast<const act_t*>(y), static_cast<const act_t*>(residual),
        static_cast<act_t*>(out), (int)s->count, s->c, s->relu, apply_reversed(s), gamma, beta,
        save_mean, save_invstd);
    return launch_check("bn_relu_fused launch");
}

int dbl_bn_relu_fused_parts(const dbl_bn_shape* s, const void* y, const float* parts, int32_t nparts,
                            const float* gamma, const float* beta, const void* residual, void* out, float* save_mean,
                            float* save_invstd, void* stream)
{
    using namespace dbl;
    int rc = check_shape(s, "bn_relu_fused_parts");
    if (rc) return rc;
    if (!y || !out || !parts || !gamma || !beta || !save_mean || !save_invstd)
        return set_error(DBL_ERR_INVALID, "bn_relu_fused_parts: null pointer");
    if (nparts <= 0) return set_error(DBL_ERR_INVALID, "bn_relu_fused_parts: no partials");
    if (!aligned16(y) || !aligned16(out) || (residual && !aligned16(residual)))
        return set_error(DBL_ERR_INVALID, "bn_relu_fused_parts: tensors must be 16-byte aligned");
    if (s->count == 0) return set_error(DBL_ERR_INVALID, "bn_relu_fused_parts: empty batch has no statistics");
    cudaStream_t st = as_stream(stream);
    if (fwd_one_launch(s->count, s->c, nparts)) {
        const int slices = s->c / kFwdSliceC;
        const int64_t blocks = (s->count + kFwdSliceRows - 1) / kFwdSliceRows, cap = 2 * sm_count() / slices;
        bn_apply_parts_kernel<<<slices * (int)std::max<int64_t>(1, std::min(blocks, cap)), kThreads, 0, st>>>(
            static_cast<const act_t*>(y), static_cast<const act_t*>(residual), static_cast<act_t*>(out), (int)s->count,
            s->c, s->relu, 1.0 / (double)s->count, s->eps, parts, nparts, gamma, beta, save_mean, save_invstd);
        return launch_check("bn_apply_parts launch");
    }
    bn_fwd_finalize_parts_kernel<<<(s->c + dbl::dev::kPartialsChannels - 1) / dbl::dev::kPartialsChannels,
                                   dbl::dev::kPartialsThreads, 0, st>>>(1.0 / (double)s->count, s->c, s->eps, parts,
                                                                   nparts, save_mean, save_invstd);
    if ((rc = launch_check("bn_fwd_finalize_parts launch"))) return rc;
    bn_apply_kernel<<<bn_grid(s->count * s->c / 8), kThreads, 2 * s->c * sizeof(float), st>>>(
        static_cast<const act_t*>(y), static_cast<const act_t*>(residual),
        static_cast<act_t*>(out), (int)s->count, s->c, s->relu, apply_reversed(s), gamma, beta,
        save_mean, save_invstd);
    return launch_check("bn_relu_fused_parts launch");
}

int dbl_maxpool_bn_relu_bwd(const dbl_bn_shape* s, int32_t n, int32_t h, int32_t w, const void* dp, const void* dp2,
                            const uint8_t* argmax, const void* x, const float* gamma, const float* beta,
                            const float* save_mean, const float* save_invstd, void* da, void* dx, float* dgamma,
                            float* dbeta, void* ws, size_t ws_bytes, void* stream)
{
    using namespace dbl;
    int rc = check_shape(s, "maxpool_bn_relu_bwd");
    if (rc) return rc;
    if (n <= 0 || h <= 0 || w <= 0 || s->count != (int64_t)n * h * w || !s->relu)
        return set_error(DBL_ERR_INVALID, "maxpool_bn_relu_bwd: shape must be [n*h*w, c] with relu set");
    if (!dp || !argmax || !x || !da || !dx || !gamma || !beta || !save_mean || !save_invstd || !dgamma || !dbeta)
        return set_error(DBL_ERR_INVALID, "maxpool_bn_relu_bwd: null pointer");
    if (!aligned16(dp) || (dp2 && !aligned16(dp2)) || !aligned16(x) || !aligned16(da) || !aligned16(dx) ||
        (reinterpret_cast<uintptr_t>(argmax) & 7))
        return set_error(DBL_ERR_INVALID, "maxpool_bn_relu_bwd: misaligned pointer");
    const size_t need = dbl_bn_workspace_bytes(s);
    if (!ws || ws_bytes < need)
        return set_error(DBL_ERR_WORKSPACE, "maxpool_bn_relu_bwd: workspace %zu < %zu bytes", ws_bytes, need);
    const int C = s->c;
    int64_t nblk = bwd_blocks(s->count, C);
    float* partial = static_cast<float*>(ws);
    float* coef = partial + nblk * 2 * C;
    cudaStream_t st = as_stream(stream);
    // small: the pool pass, then the backward in one launch (above 1024 channels the sums' staging and the
    // channel constants do not fit in 48 KB of shared memory)
    if (bwd_cluster(s->count, C, false) || C > 1024) {
        if ((rc = dbl_maxpool_bwd(n, h, w, C, dp, dp2, argmax, da, stream))) return rc;
        return bwd_launch(s, da, nullptr, x, nullptr, gamma, beta, save_mean, save_invstd, dx, nullptr, dgamma, dbeta,
                          partial, coef, nblk, st);
    }
    nblk = std::min(nblk, kPoolParts);
    bn_pool_bwd_reduce_kernel<<<reduce_grid(nblk), kPoolThreads, 3 * C * sizeof(float), st>>>(
        static_cast<const act_t*>(dp), static_cast<const act_t*>(dp2), argmax, static_cast<const act_t*>(x), n, h, w, C,
        gamma, beta, save_mean, save_invstd, (int)nblk, partial, static_cast<act_t*>(da));
    if ((rc = launch_check("bn_pool_bwd_reduce launch"))) return rc;
    return bwd_finish<kMaskY>(s, da, nullptr, x, nullptr, gamma, beta, save_mean, save_invstd, dx, dgamma, dbeta,
                              partial, coef, nblk, st);
}

size_t dbl_bn_workspace_bytes(const dbl_bn_shape* s)
{
    if (!s || s->c <= 0) return 0;
    return sizeof(float) * ((size_t)bwd_blocks(s->count, s->c) * 2 * s->c + 3 * (size_t)s->c);
}

int dbl_bn_relu_fused_bwd(const dbl_bn_shape* s, const void* dout, const void* dout2, const void* y, const void* out,
                          const float* gamma, const float* beta, const float* save_mean, const float* save_invstd, void* dy,
                          void* dresidual, float* dgamma, float* dbeta, void* ws, size_t ws_bytes, void* stream)
{
    using namespace dbl;
    int rc = check_shape(s, "bn_relu_fused_bwd");
    if (rc) return rc;
    if (!dout || !y || !dy || !gamma || !save_mean || !save_invstd || !dgamma || !dbeta || (s->relu && !out && !beta))
        return set_error(DBL_ERR_INVALID, "bn_relu_fused_bwd: null pointer");
    if (!aligned16(dout) || !aligned16(y) || !aligned16(dy) || (dout2 && !aligned16(dout2)) ||
        (out && !aligned16(out)) || (dresidual && !aligned16(dresidual)))
        return set_error(DBL_ERR_INVALID, "bn_relu_fused_bwd: tensors must be 16-byte aligned");
    if (s->count == 0) return set_error(DBL_ERR_INVALID, "bn_relu_fused_bwd: empty batch");
    const size_t need = dbl_bn_workspace_bytes(s);
    if (!ws || ws_bytes < need)
        return set_error(DBL_ERR_WORKSPACE, "bn_relu_fused_bwd: workspace %zu < %zu bytes", ws_bytes, need);
    const int C = s->c;
    const int64_t nblk = bwd_blocks(s->count, s->c);
    float* partial = static_cast<float*>(ws);
    float* coef = partial + nblk * 2 * C;
    cudaStream_t st = as_stream(stream);
    return bwd_launch(s, dout, dout2, y, out, gamma, beta, save_mean, save_invstd, dy, dresidual, dgamma, dbeta,
                      partial, coef, nblk, st);
}

}  // extern "C"

// ----------------------------------------------------------------------------- workspace-free variant
// For callers that cannot pass a workspace (see dbl_bn_relu_fused_bwd_noalloc
// in dbl.h): the per-CTA partials and the per-channel coefficients live in
// one file-scope device array sized for the largest channel count accepted.
namespace {

constexpr int kNoallocMaxBlocks = 512;  // bwd_blocks() never exceeds this
constexpr size_t kNoallocFloats =
    (size_t)kNoallocMaxBlocks * 2 * DBL_BN_NOALLOC_MAX_C + 3 * (size_t)DBL_BN_NOALLOC_MAX_C;

static __device__ __align__(256) float g_bn_noalloc_scratch[kNoallocFloats];

// Device address of the array in the calling thread's current context.  It is
// looked up (cudaGetSymbolAddress) the first time a context calls, and cached
// under that context's unique ID: a context destroyed and created again
// (cudaDeviceReset) loads the library's module again, the array may move, and
// the new ID forces a fresh lookup.  A lookup may load the module, which must
// not happen inside a stream capture, so a first call while `st` is capturing
// is refused.  (In host code the array's name is only a stand-in, never a
// device address.)
float* noalloc_scratch(cudaStream_t st, int* rc)
{
    struct Entry {
        unsigned long long ctx;
        float* ptr;
    };
    static std::mutex mu;
    static Entry cache[64] = {};
    static int used = 0;
    unsigned long long ctx = 0;
    if ((*rc = dbl::current_context_id(&ctx))) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; ctx && i < used; ++i)
        if (cache[i].ctx == ctx) {
            *rc = DBL_OK;
            return cache[i].ptr;
        }
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        (void)cudaGetLastError();
        *rc = dbl::set_error(DBL_ERR_INVALID,
                             "bn_bwd_noalloc: the first call in a CUDA context looks up the static scratch and "
                             "must come before any stream capture; call it once outside capture first");
        return nullptr;
    }
    void* p = nullptr;
    if ((*rc = dbl::cuda_check(cudaGetSymbolAddress(&p, g_bn_noalloc_scratch), "bn_bwd_noalloc: cudaGetSymbolAddress")))
        return nullptr;
    if (!ctx && (*rc = dbl::current_context_id(&ctx))) return nullptr;  // the lookup made the context current
    if (ctx && used < 64) cache[used++] = Entry{ctx, static_cast<float*>(p)};  // beyond 64 contexts: no cache
    *rc = DBL_OK;
    return static_cast<float*>(p);
}

}  // namespace

extern "C" int dbl_bn_relu_fused_bwd_noalloc(const dbl_bn_shape* s, const void* dout, const void* dout2,
                                              const void* y, const void* out, const float* gamma, const float* beta,
                                              const float* save_mean, const float* save_invstd, void* dy,
                                              void* dresidual, float* dgamma, float* dbeta, void* stream)
{
    using namespace dbl;
    int rc = check_shape(s, "bn_relu_fused_bwd_noalloc");
    if (rc) return rc;
    if (s->c > DBL_BN_NOALLOC_MAX_C)
        return set_error(DBL_ERR_UNSUPPORTED,
                         "bn_relu_fused_bwd_noalloc: %d channels exceed the static scratch limit of %d", s->c,
                         DBL_BN_NOALLOC_MAX_C);
    if (!dout || !y || !dy || !gamma || !save_mean || !save_invstd || !dgamma || !dbeta || (s->relu && !out && !beta))
        return set_error(DBL_ERR_INVALID, "bn_relu_fused_bwd_noalloc: null pointer");
    if (!aligned16(dout) || !aligned16(y) || !aligned16(dy) || (dout2 && !aligned16(dout2)) ||
        (out && !aligned16(out)) || (dresidual && !aligned16(dresidual)))
        return set_error(DBL_ERR_INVALID, "bn_relu_fused_bwd_noalloc: tensors must be 16-byte aligned");
    if (s->count == 0) return set_error(DBL_ERR_INVALID, "bn_relu_fused_bwd_noalloc: empty batch");
    const int C = s->c;
    const int64_t nblk = bwd_blocks(s->count, s->c);
    if (nblk > kNoallocMaxBlocks || (size_t)nblk * 2 * C + 3 * (size_t)C > kNoallocFloats)
        return set_error(DBL_ERR_UNSUPPORTED, "bn_relu_fused_bwd_noalloc: shape exceeds the static scratch");
    cudaStream_t st = as_stream(stream);
    float* partial = noalloc_scratch(st, &rc);
    if (rc) return rc;
    float* coef = partial + nblk * 2 * C;  // written by the finalize kernel before the apply kernel reads it
    return bwd_launch(s, dout, dout2, y, out, gamma, beta, save_mean, save_invstd, dy, dresidual, dgamma, dbeta,
                      partial, coef, nblk, st);
}
