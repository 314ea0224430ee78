// conv.cu -- convolution forward, data-gradient and weight-gradient passes of
// ResNet-18 (Sec. 5.1.1; the gradients are those of the batch-mean loss of
// Eq. 1) as implicit GEMMs on the sm_103a tensor cores.
//
// conv_igemm_kernel serves every pass; conv_splitk_kernel is its form for shapes with fewer tiles than
// CTA pairs, and the window, pixel-pair, row-block and filter-row kernels further down replace it
// where a stride-1 pass can read shifted rows of one strip.  A CTA owns a 128 x BN tile of the
// GEMM result D, accumulated in tensor memory (TMEM) by tcgen05.mma with bf16
// operands and fp32 accumulation:
//
//   pass   D rows (M)          D cols (N)     reduction            A operand            B operand
//   fwd    output pixels n,p,q out channel k  taps x in channels   im2col(x), K-major   w [k][rsc], K-major
//   dgrad  input pixels n,h,w  in channel c   taps x out channels  im2col(dy), K-major  w [k][rs][c], MN-major
//   wgrad  taps x in channel   out channel k  output pixels        im2col(x), MN-major  dy [pix][k], MN-major
//
// Operands are staged in shared memory by TMA: the activation side with
// im2col-mode tensor maps (the bounding box handles zero padding, stride and
// the ragged tail of the last tile), the other side with tiled tensor maps,
// all with 128-byte swizzling (no swizzle for the 8-channel stem input).
// Warp roles: two producer warps issue TMA loads into a ring of stages guarded by
// full/empty mbarriers, one warp allocates TMEM and issues the MMAs (one thread), and
// the first four or eight warps drain TMEM to global memory (bf16 rows plus BatchNorm
// channel statistics for fwd, fp32 split-K partials for wgrad).
//
// Stride-2 data gradients are split into the 4 output phases (h mod 2,
// w mod 2); each phase is a stride-1 correlation with the taps of matching
// parity, so no MMA work is spent on the zeros of the strided input.
// Every mbarrier wait is bounded (see dbl_internal.cuh); a wait that gives up
// records DBL_ERR_TIMEOUT in the device status word and the CTA winds down.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include <atomic>

#include "dbl_internal.cuh"

namespace {

using namespace dbl::dev;

constexpr int BM = 128;        // tile rows = TMEM lanes

enum Mode : int { kFwd = 0, kDgrad = 1, kWgrad = 2, kFwdC8 = 3, kWgradC8 = 4 };

__device__ int g_conv_status;  // DBL_OK or DBL_ERR_TIMEOUT, read by dbl_device_status()

constexpr int kMaxGrid = 256;     // persistent grid never exceeds this (workspace sizing)
constexpr int kMaxNcols = 512;    // widest D (output channels of ResNet-18)

struct ConvParams {
    int mode;
    int M;              // D rows (for dgrad: rows of one phase)
    int Ncols;          // D columns
    int m_tiles, n_tiles, zdim;  // tile grid; zdim = split-K slices (wgrad) or phases (dgrad)
    int total_tiles;
    // traversal grid of the im2col operand: (images, rows, cols) and origin of grid point (0,0)
    int gN, gP, gQ;
    int tstride_h, tstride_w;  // origin step per grid step
    int base_h, base_w;
    int cblocks;        // 64-channel blocks in the reduction (fwd: C/64, dgrad: K/64)
    int ntaps;          // R*S
    int S;              // filter width
    int Cin;            // input channels (fwd B column offset, wgrad row -> (tap, c))
    int num_kb;         // K-blocks of the whole reduction (fwd, wgrad); per phase from the table (dgrad)
    int kb_per_split;   // wgrad split-K chunk
    // dgrad phase tables
    int phase_div;      // 1 or 2
    int out_h, out_w;   // full dx spatial size
    int phase_off[5];
    int8_t tap_r[16], tap_s[16], tap_oh[16], tap_ow[16];
    int proj_kb;        // dgrad phase (0,0): extra K-blocks of a 1x1 stride-2 projection's dy2 . w2
    // outputs
    void* out;          // bf16 rows (fwd, dgrad); fp32 dw (wgrad, one slice) or fp32 slices [z][Ncols][M]
    int64_t ldo;        // elements between output rows (fwd, dgrad)
    int st32;           // 16-bit outputs whose base and row pitch are multiples of 32 bytes: 32-byte stores
    int wg_accumulate;  // wgrad with one slice: add into dw
    float* stats;       // fwd: [gridDim.x][2][Ncols] per-CTA channel sums, or nullptr
    // window kernel (3x3, stride 1, pad 1): the batch as one column of zero-padded images
    int win_R, win_S;         // filter taps along H and W
    int win_ph, win_pw;       // padding along H and W (a strip row copy starts at column -pw)
    int win_P, win_Q;         // output height and width: positions with h < P, w < Q are outputs
    int win_Hp, win_Wp;       // padded height and width (H + 2*ph, W + 2*pw)
    int win_tile;             // positions per tile (weight gradient: per K-block), <= 256
    int win_srows;            // padded rows loaded per strip (weight gradient: x strip)
    int win_dyrows;           // weight gradient: padded rows of the dy strip
    int win_strip_bytes;      // bytes of one strip buffer, or of one x + dy stage (a multiple of 1024)
    int win_margin;           // CTA pairs: bytes before and after each strip buffer (0 for single CTAs);
                              // row-block weight gradient: offset of the dy strip in a stage
    int win_stages;           // row-block weight gradient: x + dy stages
    int win_bpi;              // row-block and filter-row weight gradient: K-blocks per image
    int win_ni;               // filter-row weight gradient: images per K-block; bands: bands per image
    int win_cl;               // filter-row weight gradient: CTAs per cluster, which add their sums on chip
    int test_stall;           // dbl_conv_test_stall_next: block 0 never loads (its part of) its first K-block
};

__device__ __forceinline__ void report_timeout(volatile int* abort)
{
    *abort = 1;
    atomicExch(&g_conv_status, DBL_ERR_TIMEOUT);
}

constexpr int kProducers = 2;     // producer warps; producer p fills the stages of iterations it % 2 == p

enum Family : int { kFamFwd = 0, kFamWgrad = 1 };  // fwd/dgrad/stem-fwd, and the two weight-gradient modes

// Per (tile width, family) geometry.  mbarrier round trips and TMA issues cost a
// thread on the order of a hundred cycles each, so every ring stage is sized to
// carry at least ~384 cycles of MMA work per handful of TMA ops:
//   forward family, BN <= 128: a tile is 256 rows in two 128-row accumulators
//     that share one B tile; one 256-pixel im2col op feeds both;
//   weight-gradient family: a K-block is 128 pixels (8 MMA K-steps).
template <int BN, int FAM, int CG = 1>
struct Cfg {
    static constexpr int ACC = (FAM == kFamFwd && BN <= 128) ? 2 : 1;  // 128-row accumulators per tile
    static constexpr int BMT = 128 * ACC;                               // tile rows per CTA
    static constexpr int KB = FAM == kFamFwd ? 64 : 128;                // reduction elements per stage
    static constexpr int KSTEPS = KB / 16;
    static constexpr int BNC = BN / CG;                                 // B columns held by one CTA
    static constexpr int A_BYTES = BMT * KB * 2;
    static constexpr int B_BYTES = BNC * KB * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int MAX_STAGES = CG == 2 ? 6 : 4;
    static constexpr int STAGES = (196608 / STAGE_BYTES) < MAX_STAGES ? (196608 / STAGE_BYTES) : MAX_STAGES;
    static constexpr int RING = STAGES * STAGE_BYTES;
    // Epilogue warps: two per TMEM lane quarter for the wider tiles, each draining half of the columns
    // (the last tile's epilogue is not hidden behind MMAs; with four warps it takes 750 cycles per 32
    // columns with channel sums): forward at 10x10x256, batch 128 20.4 -> 18.5 us, 7x7x512, batch 128
    // 30.1 -> 28.2, its data gradient 27.5 -> 27.2; a 14x14 1x1 projection 256 -> 512 11.5 -> 9.8
    // (weight gradients keep four, whose CTAs start sooner: 4x4 maps of 256 channels, one image 8.2 us with eight and
    // 7.7 with four, 3x3 maps 128 -> 256, batch 16 8.8 and 8.4)
    static constexpr int EPI = BN > 64 && FAM == kFamFwd ? 8 : 4;
    static constexpr int CW = BN * 4 / EPI;                    // columns one epilogue warp drains
    static constexpr int EPI_TILE = BN > 64 ? 0 : 4 * 32 * 33 * 4;  // per-warp 32x32 transpose scratch (RowStats)
    static constexpr int EPI_SUM = 4 * 2 * kMaxNcols * 4;      // channel sums per lane quarter (fwd)
    static constexpr int SMEM = RING + EPI_TILE + EPI_SUM + 1024;  // + 1 KB alignment slack
    static constexpr int NB = ACC * BN <= 128 ? 4 : 2;          // tiles in flight (TMEM accumulator buffers)
    static constexpr uint32_t TMEM_COLS = NB * ACC * BN;
    static constexpr int THREADS = 32 * (EPI + kProducers + 1);  // epilogue, producers, MMA
    static constexpr int MMA_WARP = EPI + kProducers;
    static_assert(STAGES >= 2, "ring too shallow");
    static_assert(TMEM_COLS <= 512, "TMEM holds 512 columns");
    static_assert(SMEM <= 232448 - 1024, "shared memory per CTA");
    static_assert(CG == 1 || SMEM >= 117 * 1024, "a cluster kernel's CTA has its SM to itself (kClusterSmem)");
};

struct TileCoord {
    int m_tile, n_tile, z;
};

// Weight gradient: split-K slice outermost, so that the CTAs running at one time
// share the slice's dy K-blocks.  Stride-2 data gradient: the four phases of one
// m-tile are adjacent, so that the dy rows they all read are fetched from DRAM
// once; the phase index is rotated by one per wave of the persistent grid, so
// that every CTA gets a mix of the 4-, 2- and 1-tap phases.
// units: the number of tiles the persistent grid processes at one time.
__device__ __forceinline__ TileCoord decode_tile(const ConvParams& p, int t, int units)
{
    TileCoord c;
    if (p.mode == kDgrad && p.zdim > 1) {
        const int g = t / p.zdim, l = t - g * p.zdim;
        const int per_wave = max(1, units / p.zdim);
        c.z = (l + g / per_wave) % p.zdim;
        c.m_tile = g / p.n_tiles;
        c.n_tile = g - c.m_tile * p.n_tiles;
        return c;
    }
    const int mn = p.m_tiles * p.n_tiles;
    c.z = t / mn;
    const int r = t - c.z * mn;
    c.m_tile = r / p.n_tiles;
    c.n_tile = r - c.m_tile * p.n_tiles;
    return c;
}

// Number of K-blocks a tile reduces, and the first one.
__device__ __forceinline__ void kb_range(const ConvParams& p, int z, int& kb0, int& nkb)
{
    if (p.mode == kDgrad) {
        kb0 = 0;
        nkb = (p.phase_off[z + 1] - p.phase_off[z]) * p.cblocks + (z == 0 ? p.proj_kb : 0);
    } else if (p.mode == kWgrad || p.mode == kWgradC8) {
        kb0 = z * p.kb_per_split;
        nkb = min(p.num_kb, kb0 + p.kb_per_split) - kb0;
        if (nkb < 0) nkb = 0;
    } else {
        kb0 = 0;
        nkb = p.num_kb;
    }
}

// Issue the TMA loads of one K-block of one tile into ring stage (sa, sb); fb is
// the shared::cluster address of the stage's full barrier.  With CTA pairs
// (CG = 2) CTA `rank` loads its own 128-row (fwd family: BMT-row) part of A and
// columns rank*BN/2 .. (rank+1)*BN/2-1 of B, and both CTAs' loads complete on
// rank 0's barrier.
template <int BN, int FAM, int CG>
__device__ __forceinline__ void load_kblock(const ConvParams& p, const CUtensorMap* tmA, const CUtensorMap* tmB,
                                            const CUtensorMap* tmA2, const CUtensorMap* tmB2, uint8_t* sa,
                                            uint8_t* sb, uint32_t fb, const TileCoord& tc, int kb, int tn, int tp,
                                            int tq, int rank)
{
    using C = Cfg<BN, FAM, CG>;
    const int64_t gPQ = (int64_t)p.gP * p.gQ;
    const int ncol0 = tc.n_tile * BN + rank * C::BNC;  // first B column this CTA loads
    if constexpr (FAM == kFamFwd) {
        if (p.mode == kFwd) {
            const int tap = kb / p.cblocks, cb = kb - tap * p.cblocks;
            const int r = tap / p.S, sx = tap - r * p.S;
            tma_load_im2col_4d_cg<CG>(sa, tmA, fb, cb * 64, tq * p.tstride_w + p.base_w, tp * p.tstride_h + p.base_h, tn,
                                      (uint16_t)sx, (uint16_t)r);
            tma_load_2d_cg<CG>(sb, tmB, fb, tap * p.Cin + cb * 64, ncol0);
        } else if (p.mode == kDgrad && kb >= (p.phase_off[tc.z + 1] - p.phase_off[tc.z]) * p.cblocks) {
            // phase (0,0) of a stride-2 data gradient with a 1x1 stride-2 projection shortcut on
            // the same input: dx[n, 2i, 2j] also receives dy2[n, i, j] . w2, the dy2 rows of this
            // tile being the tile's own rows m0.. (tmA2: dy2 as [n*P*Q][k2], tmB2: w2 as [k2][1][c])
            const int e = kb - (p.phase_off[tc.z + 1] - p.phase_off[tc.z]) * p.cblocks;
            const int m0 = (tn * p.gP + tp) * p.gQ + tq;
            tma_load_2d_cg<CG>(sa, tmA2, fb, e * 64, m0);
            for (int j = 0; j < C::BNC / 64; ++j) tma_load_3d_cg<CG>(sb + j * 8192, tmB2, fb, ncol0 + 64 * j, 0, e * 64);
        } else if (p.mode == kDgrad) {
            const int t = p.phase_off[tc.z] + kb / p.cblocks, kbk = kb % p.cblocks;
            tma_load_im2col_4d_cg<CG>(sa, tmA, fb, kbk * 64, tq + p.base_w, tp + p.base_h, tn, (uint16_t)p.tap_ow[t],
                                      (uint16_t)p.tap_oh[t]);
            const int wtap = p.tap_r[t] * p.S + p.tap_s[t];
            for (int j = 0; j < C::BNC / 64; ++j)
                tma_load_3d_cg<CG>(sb + j * 8192, tmB, fb, ncol0 + 64 * j, wtap, kbk * 64);
        } else {  // kFwdC8: 8 taps of 8 channels; taps past R*S read a valid tap and meet zero weights
            for (int j = 0; j < 8; ++j) {
                int tap = kb * 8 + j;
                const int wcol = tap * 8;
                if (tap >= p.ntaps) tap = p.ntaps - 1;
                tma_load_im2col_4d_cg<CG>(sa + j * (C::BMT * 16), tmA, fb, 0, tq * p.tstride_w + p.base_w,
                                          tp * p.tstride_h + p.base_h, tn, (uint16_t)(tap % p.S), (uint16_t)(tap / p.S));
                tma_load_2d_cg<CG>(sb + j * (C::BNC * 16), tmB, fb, wcol, ncol0);
            }
        }
    } else {
        // weight gradient: a K-block is 128 output pixels
        const int64_t pix0 = (int64_t)kb * 128;
        const int n = (int)(pix0 / gPQ);
        const int64_t rem = pix0 - (int64_t)n * gPQ;
        const int pp = (int)(rem / p.gQ), qq = (int)(rem - (int64_t)pp * p.gQ);
        if (p.mode == kWgrad) {
            for (int h = 0; h < 2; ++h) {
                const int mrow = (tc.m_tile * CG + rank) * BM + 64 * h;
                int tap = mrow / p.Cin;
                const int c0 = mrow - tap * p.Cin;
                if (tap >= p.ntaps) tap = 0;  // rows past R*S*C: loaded, never stored
                tma_load_im2col_4d_cg<CG>(sa + h * 16384, tmA, fb, c0, qq * p.tstride_w + p.base_w,
                                          pp * p.tstride_h + p.base_h, n, (uint16_t)(tap % p.S), (uint16_t)(tap / p.S));
            }
        } else {  // kWgradC8: 16 taps x 8 channels of rows
            for (int j = 0; j < 16; ++j) {
                int tap = tc.m_tile * 16 + j;
                if (tap >= p.ntaps) tap = 0;
                tma_load_im2col_4d_cg<CG>(sa + j * 2048, tmA, fb, 0, qq * p.tstride_w + p.base_w,
                                          pp * p.tstride_h + p.base_h, n, (uint16_t)(tap % p.S), (uint16_t)(tap / p.S));
            }
        }
        for (int j = 0; j < C::BNC / 64; ++j) tma_load_2d_cg<CG>(sb + j * 16384, tmB, fb, ncol0 + 64 * j, (int)pix0);
    }
}

// Epilogue of the 16-bit-output passes for one 32-column chunk of this thread's
// accumulator row: round to the storage format (bf16, or f16) and store the row chunk (if the row is a real
// output); back[] receives the stored values (zeros for rows that are not outputs).
__device__ __forceinline__ void store_row_chunk_act(const ConvParams& p, const uint32_t (&v)[32], bool valid,
                                                     int64_t out_row, int col0, float (&back)[32])
{
    uint4 pk[4];
    uint32_t* w32 = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t u = valid ? dbl::act::pack2_u32(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1]))
                                 : 0u;  // rows that are not outputs: 0
        w32[k] = u;
        const float2 f = dbl::act::unpack2_u32(u);  // the stored values (16-bit -> fp32 is exact)
        back[2 * k] = f.x;
        back[2 * k + 1] = f.y;
    }
    if (valid) {
        act_t* o = static_cast<act_t*>(p.out) + out_row * p.ldo + col0;
        if (p.st32) {
            // whole 32-byte sectors per instruction: half the store instructions and L2 write
            // requests of 16-byte stores, each of which fills half a sector
#pragma unroll
            for (int k = 0; k < 2; ++k)
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o + 16 * k),
                             "r"(pk[2 * k].x), "r"(pk[2 * k].y), "r"(pk[2 * k].z), "r"(pk[2 * k].w),
                             "r"(pk[2 * k + 1].x), "r"(pk[2 * k + 1].y), "r"(pk[2 * k + 1].z), "r"(pk[2 * k + 1].w)
                             : "memory");
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) reinterpret_cast<uint4*>(o)[k] = pk[k];
        }
    }
}

// BatchNorm channel sums (sum y, sum y^2) of the stored forward outputs, kept
// in registers across the tiles of a CTA instead of being reduced across the
// warp for every tile (which costs shared-memory bandwidth that the mainloop
// needs).  Thread (warp, lane) adds the values of its own accumulator row.
// flush() reduces over the lanes through the warp's 32x33 scratch and adds the
// column totals to the warp's channel sums (once per CTA).
template <int BN>
struct RowStats {
    static constexpr int NCH = BN / 32;
    float s[NCH][32], q[NCH][32];

    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int c = 0; c < NCH; ++c)
#pragma unroll
            for (int k = 0; k < 32; ++k) s[c][k] = q[c][k] = 0.f;
    }

    // x: the stored values of chunk ch of this thread's row (call with ch a compile-time
    // constant after unrolling); the sum of squares by fused multiply-add.
    __device__ __forceinline__ void add(int ch, const float (&x)[32])
    {
#pragma unroll
        for (int k = 0; k < 32; k += 2) {
            const float2 v = make_float2(x[k], x[k + 1]);
            const float2 a = add2(make_float2(s[ch][k], s[ch][k + 1]), v);
            const float2 b = fma2(v, v, make_float2(q[ch][k], q[ch][k + 1]));
            s[ch][k] = a.x;
            s[ch][k + 1] = a.y;
            q[ch][k] = b.x;
            q[ch][k + 1] = b.y;
        }
    }

    // wsum: [2][ncols] channel sums; col_base: the warp's first column.
    __device__ __forceinline__ void flush(float* st_tile, float* wsum, int ncols, int col_base, int lane)
    {
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
#pragma unroll
            for (int w = 0; w < 2; ++w) {
#pragma unroll
                for (int k = 0; k < 32; ++k) st_tile[lane * 33 + k] = w ? q[c][k] : s[c][k];
                __syncwarp();
                float tot = 0.f;
#pragma unroll
                for (int u = 0; u < 32; ++u) tot += st_tile[u * 33 + lane];
                __syncwarp();
                wsum[w * ncols + col_base + c * 32 + lane] += tot;
            }
        }
        zero();
    }
};

// The same sums for tiles of 128 and 256 columns, without shuffles per tile: the accumulator is read a
// second time in the 16x256b layout (tmem_ld_16x256b_x4), in which a thread holds 4 of the warp's 32
// rows at 8 of each 32 columns, and rounds them to the storage format as the store does.  flush()
// adds the eight lanes that share columns (seven shuffles per array of eight), once per CTA.  RowStats
// at these widths spends about 300 instructions, 32 to 48 of them shuffles, per 32 x 32 chunk against
// about 130 here, which one-tile CTAs cannot hide: forward at 28x28x128, batch 512 87.0 -> 80.4 us,
// 7x7x512, batch 128 32.2 -> 30.1, a 20x20 1x1 projection 128 -> 256, batch 128 12.3 -> 10.9 (without
// channel sums 74.1, 27.2 and 8.1).
template <int BN>
struct ColStats {
    static constexpr int NCH = BN / 32;
    float2 s[NCH][4], q[NCH][4];  // [chunk][group]: columns 8*group + 2*(lane%4), + 1

    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int c = 0; c < NCH; ++c)
#pragma unroll
            for (int g = 0; g < 4; ++g) s[c][g] = q[c][g] = make_float2(0.f, 0.f);
    }

    // lo, hi: rows 0-15 and 16-31 of chunk ch; valid: bit i = row i is an output.
    __device__ __forceinline__ void add(int ch, const uint32_t (&lo)[16], const uint32_t (&hi)[16], uint32_t valid,
                                        int lane)
    {
        const uint32_t v = valid >> (lane / 4);
        const bool ok[4] = {(v & 1u) != 0, (v & 0x100u) != 0, (v & 0x10000u) != 0, (v & 0x1000000u) != 0};
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float2 f[4];  // rows lane/4, +8, +16, +24
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const uint32_t a = h < 2 ? lo[4 * g + 2 * h] : hi[4 * g + 2 * (h - 2)];
                const uint32_t b = h < 2 ? lo[4 * g + 2 * h + 1] : hi[4 * g + 2 * (h - 2) + 1];
                f[h] = dbl::act::unpack2_u32(ok[h] ? dbl::act::pack2_u32(__uint_as_float(a), __uint_as_float(b)) : 0u);
            }
            s[ch][g] = add2(s[ch][g], add2(add2(f[0], f[1]), add2(f[2], f[3])));
            q[ch][g] = add2(q[ch][g], add2(fma2(f[0], f[0], mul2(f[1], f[1])), fma2(f[2], f[2], mul2(f[3], f[3]))));
        }
    }

    // Sum over the eight lanes that share columns: three steps that halve the values a lane keeps;
    // returns value k (see flush) of 2*group + e.
    __device__ __forceinline__ static float fold(const float2 (&f)[4], int lane)
    {
        const bool b16 = (lane & 16) != 0, b8 = (lane & 8) != 0, b4 = (lane & 4) != 0;
        float2 h[2];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const float2 send = b16 ? f[g] : f[g + 2], keep = b16 ? f[g + 2] : f[g];
            h[g].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 16);
            h[g].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 16);
        }
        const float2 send = b8 ? h[0] : h[1], keep = b8 ? h[1] : h[0];
        const float x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 8);
        const float y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 8);
        return (b4 ? y : x) + __shfl_xor_sync(0xffffffffu, b4 ? x : y, 4);
    }

    __device__ __forceinline__ void flush(float* wsum, int ncols, int col_base, int lane)
    {
        const int k = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);  // the value this lane keeps
        float* dst = wsum + col_base + 8 * (k >> 1) + 2 * (lane & 3) + (k & 1);
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            dst[c * 32] += fold(s[c], lane);
            dst[ncols + c * 32] += fold(q[c], lane);
        }
        __syncwarp();
        zero();
    }
};

// The statistics of an epilogue warp of a BN-column tile: ColStats over half of the columns, or RowStats.
template <int BN>
using TileStats = std::conditional_t<(BN > 64), ColStats<BN / 2>, RowStats<BN>>;

// Persistent kernel: CTA b processes tiles b, b + gridDim.x, ...  The ring of
// STAGES shared-memory stages runs continuously across tiles; two producer
// warps fill alternate stages; two TMEM accumulators let the epilogue of one
// tile overlap the MMAs of the next.
//
// CG = 2 (clusters of two CTAs): a tile is processed by a CTA pair with
// M = 256 MMAs (tcgen05 .cta_group::2).  Each CTA stages its own BMT rows of A
// and half of the B columns, so a CTA's shared memory carries half of the B
// bytes (TMA writes and MMA reads) of the single-CTA form; shared-memory
// bandwidth is what limits the single-CTA form.  Rank 0 issues the MMAs and owns
// the stage-full barriers, which both CTAs' loads complete on; its commits
// arrive on the stage-empty and accumulator-full barriers of both CTAs; the
// epilogues of both CTAs arrive on rank 0's accumulator-empty barriers.  Each
// CTA drains its own TMEM (its own rows, all BN columns).
template <int BN, int FAM, int CG>
__global__ void __launch_bounds__(Cfg<BN, FAM, CG>::THREADS, 1)
    conv_igemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
                      const ConvParams p)
{
    using C = Cfg<BN, FAM, CG>;
    constexpr int STAGES = C::STAGES;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], accf_bar[C::NB], acce_bar[C::NB], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    float* epi_tile = reinterpret_cast<float*>(sgen + C::RING);
    float* epi_sum = reinterpret_cast<float*>(sgen + C::RING + C::EPI_TILE);
    const int rank = CG == 2 ? (int)cluster_ctarank() : 0;
    const int unit0 = blockIdx.x / CG, nunits = gridDim.x / CG;  // this pair's first tile, tiles' stride

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < C::NB; ++b) {
            mbar_init(&accf_bar[b], 1);
            mbar_init(&acce_bar[b], C::EPI * CG);  // one arrival per epilogue warp of the pair
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    const bool want_stats = FAM == kFamFwd && (p.mode == kFwd || p.mode == kFwdC8) && p.stats != nullptr;
    if (want_stats)
        for (int i = threadIdx.x; i < 4 * 2 * p.Ncols; i += blockDim.x) epi_sum[i] = 0.f;
    if (warp >= C::EPI && warp < C::MMA_WARP && lane == 0) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        if (p.proj_kb) {
            tma_prefetch_desc(&tmA2);
            tma_prefetch_desc(&tmB2);
        }
    }
    if (warp == C::MMA_WARP) {
        tmem_alloc_cg<CG>(&tmem_slot, C::TMEM_COLS);
        tmem_relinquish_cg<CG>();
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) cluster_sync_all();  // both CTAs' barriers initialised, TMEM allocated
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;
    const int64_t gPQ = (int64_t)p.gP * p.gQ;

    if (warp >= C::EPI && warp < C::MMA_WARP) {
        // ------------------------------------------------------------------ TMA producers (whole warp, one lane issues)
        const int prod = warp - C::EPI;
        int it = 0, last_it = -1;
        bool failed = false;
        for (int t = unit0; t < p.total_tiles; t += nunits) {
            const TileCoord tc = decode_tile(p, t, nunits);
            int kb0, nkb;
            kb_range(p, tc.z, kb0, nkb);
            int tn = 0, tp = 0, tq = 0;
            if (FAM == kFamFwd) {
                const int64_t m0 = ((int64_t)tc.m_tile * CG + rank) * C::BMT;
                tn = (int)(m0 / gPQ);
                const int64_t rem = m0 - (int64_t)tn * gPQ;
                tp = (int)(rem / p.gQ);
                tq = (int)(rem - (int64_t)tp * p.gQ);
            }
            for (int k = 0; k < nkb; ++k, ++it) {
                if (it % kProducers != prod) continue;
                if (p.test_stall && blockIdx.x == 0 && it == 0) continue;  // stage 0 never fills (bounded-wait test)
                const int s = it % STAGES;
                const uint32_t ok = mbar_wait_warp(&empty_bar[s], ((it / STAGES) & 1) ^ 1, &abort_flag);
                if (__any_sync(0xffffffffu, ok == 0u)) {
                    failed = true;
                    break;
                }
                uint8_t* sa = sgen + s * C::STAGE_BYTES;
                uint32_t fb = smem_u32(&full_bar[s]);
                if (CG == 1 || rank == 0)
                    mbar_arrive_expect_tx_elect(&full_bar[s], (uint32_t)(CG * C::STAGE_BYTES));
                if (CG == 2) fb = mapa_shared(fb, 0);
                load_kblock<BN, FAM, CG>(p, &tmA, &tmB, &tmA2, &tmB2, sa, sa + C::A_BYTES, fb, tc, kb0 + k, tn, tp, tq,
                                         rank);
                last_it = it;
            }
            if (failed) break;
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            if (CG == 1 || rank == 0) {
                // let copies this producer issued land before the CTA's shared memory goes away
                for (int i = last_it; i >= 0 && i > last_it - STAGES * kProducers; i -= kProducers)
                    (void)mbar_drain_warp(&full_bar[i % STAGES], (i / STAGES) & 1);
            } else {
                // rank 1's copies complete on rank 0's barriers: give them a fixed time instead
                const uint64_t t0 = globaltimer();
                while (globaltimer() - t0 < 1000000ull) {
                }
            }
        }
    } else if (warp == C::MMA_WARP) {
        // ------------------------------------------------------------------ MMA issuer (whole warp, one lane issues)
        const bool a_mn = (p.mode == kWgrad || p.mode == kWgradC8);
        const bool b_mn = (p.mode != kFwd && p.mode != kFwdC8);
        const uint32_t idesc = idesc_act(BM * CG, BN, a_mn ? 1u : 0u, b_mn ? 1u : 0u);
        constexpr uint16_t kAll = CG == 2 ? 3 : 1;  // commits reach both CTAs of a pair
        // Operand descriptors without their start address, and the start-address steps
        // (in 16-byte units) per K-step and per accumulator:
        //   kFwd / kDgrad: A K-major, 128-byte swizzle, one K-step = 32 bytes of a row;
        //     B K-major (fwd) or MN-major with 64-wide atoms 8 KB apart (dgrad, 2 KB per K-step);
        //   kFwdC8: K-major without swizzle: core matrices of 8 rows x 16 B, rows 16 B apart,
        //     8-row groups 128 B apart (SBO), the two taps of one K-step LBO apart;
        //   kWgrad: both MN-major, 128-byte swizzle, 64-wide atoms 16 KB apart (LBO);
        //   kWgradC8: A MN-major without swizzle, 8 pixels x 8 channels per core matrix,
        //     next 8 pixels 128 B apart (LBO), next tap 2 KB apart (SBO).
        uint64_t dA, dB;
        int a_step16, b_step16, a_acc16 = 16384 / 16;
        if (p.mode == kFwd || p.mode == kDgrad) {
            dA = smem_desc(0, 16, 1024, kSwizzle128B);
            a_step16 = 2;
            if (p.mode == kFwd) {
                dB = smem_desc(0, 16, 1024, kSwizzle128B);
                b_step16 = 2;
            } else {
                dB = smem_desc(0, 8192, 1024, kSwizzle128B);
                b_step16 = 2048 / 16;
            }
        } else if (p.mode == kFwdC8) {
            dA = smem_desc(0, C::BMT * 16, 128, kSwizzleNone);
            dB = smem_desc(0, C::BNC * 16, 128, kSwizzleNone);
            a_step16 = 2 * C::BMT;
            b_step16 = 2 * C::BNC;
            a_acc16 = 2048 / 16;
        } else if (p.mode == kWgrad) {
            dA = smem_desc(0, 16384, 1024, kSwizzle128B);
            dB = smem_desc(0, 16384, 1024, kSwizzle128B);
            a_step16 = b_step16 = 2048 / 16;
        } else {
            dA = smem_desc(0, 128, 2048, kSwizzleNone);
            dB = smem_desc(0, 16384, 1024, kSwizzle128B);
            a_step16 = 256 / 16;
            b_step16 = 2048 / 16;
        }
        // The MMA issue is on the critical path: every cycle this warp spends polling a
        // barrier while the tensor pipe has nothing queued is lost.  So the wait for the next
        // stage is made before the last K-step of the current stage is issued, while the
        // tensor pipe still has work.
        bool failed = false;
        auto wait_ok = [&](uint64_t* bar, uint32_t parity) -> bool {
            const uint32_t ok = mbar_wait_warp(bar, parity, &abort_flag);
            return !__any_sync(0xffffffffu, ok == 0u);
        };
        // Only waits inside a tile are made ahead: waiting for the next tile's accumulator or
        // data before this tile's last K-step would delay this tile's completion, and with it
        // the epilogue, behind an earlier epilogue or a later load.
        int it = 0, lt = 0;
        for (int t = unit0; t < p.total_tiles && (CG == 1 || rank == 0) && !failed; t += nunits, ++lt) {
            const TileCoord tc = decode_tile(p, t, nunits);
            int kb0, nkb;
            kb_range(p, tc.z, kb0, nkb);
            const int buf = lt % C::NB;
            if (!wait_ok(&acce_bar[buf], ((lt / C::NB) & 1) ^ 1) ||
                (nkb > 0 && !wait_ok(&full_bar[it % STAGES], (it / STAGES) & 1))) {
                failed = true;
                break;
            }
            const uint32_t d = tmem + (uint32_t)(buf * C::ACC * BN);
            for (int k = 0; k < nkb; ++k, ++it) {
                tc_fence_after();
                const int s = it % STAGES;
                const uint32_t sa = sbase + s * C::STAGE_BYTES;
                const uint32_t sb = sa + C::A_BYTES;
                const uint64_t ad0 = dA | (uint64_t)((sa >> 4) & 0x3FFFu), bd0 = dB | (uint64_t)((sb >> 4) & 0x3FFFu);
#pragma unroll
                for (int j = 0; j < C::KSTEPS - 1; ++j) {
#pragma unroll
                    for (int a = 0; a < C::ACC; ++a)
                        mma_act_elect_cg<CG>(d + a * BN, ad0 + (uint64_t)(a * a_acc16 + j * a_step16),
                                              bd0 + (uint64_t)(j * b_step16), idesc, (k > 0 || j > 0) ? 1u : 0u);
                }
                if (k + 1 < nkb) failed = !wait_ok(&full_bar[(it + 1) % STAGES], ((it + 1) / STAGES) & 1);
                constexpr int jl = C::KSTEPS - 1;
#pragma unroll
                for (int a = 0; a < C::ACC; ++a)
                    mma_act_elect_cg<CG>(d + a * BN, ad0 + (uint64_t)(a * a_acc16 + jl * a_step16),
                                          bd0 + (uint64_t)(jl * b_step16), idesc, (k > 0 || jl > 0) ? 1u : 0u);
                mma_commit_elect_cg<CG>(&empty_bar[s], kAll);
                if (failed) {
                    ++it;
                    break;
                }
            }
            mma_commit_elect_cg<CG>(&accf_bar[buf], kAll);  // arrives when this tile's MMAs have completed
        }
        if (failed && lane == 0) report_timeout(&abort_flag);
        if (CG == 1 || rank == 0) {
            // every MMA issued above completes before the accumulators are freed
            mma_commit_elect_cg<CG>(&drain_bar, 1);
            (void)mbar_drain_warp(&drain_bar, 0);
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 0 .. EPI-1)
        constexpr int CW = C::CW, NCH = CW / 32;
        const int quarter = warp & 3, cw0 = (warp >> 2) * CW;  // TMEM lanes 32*quarter.., tile columns cw0..
        [[maybe_unused]] float* st_tile = epi_tile + warp * 32 * 33;
        float* wsum = epi_sum + quarter * 2 * p.Ncols;
        TileStats<BN> rs;
        rs.zero();
        auto flush = [&](int ntile) {
            if constexpr (BN > 64)
                rs.flush(wsum, p.Ncols, ntile * BN + cw0, lane);
            else
                rs.flush(st_tile, wsum, p.Ncols, ntile * BN, lane);
        };
        int stats_ntile = -1;  // column tile the register sums belong to
        int lt = 0;
        for (int t = unit0; t < p.total_tiles; t += nunits, ++lt) {
            const TileCoord tc = decode_tile(p, t, nunits);
            int kb0, nkb;
            kb_range(p, tc.z, kb0, nkb);
            const int buf = lt % C::NB;
            const uint32_t ok = mbar_wait_warp(&accf_bar[buf], (lt / C::NB) & 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                if (lane == 0) report_timeout(&abort_flag);
                break;
            }
            tc_fence_after();
            const int row = quarter * 32 + lane;  // TMEM lane = row within a 128-row accumulator
            const bool have_acc = nkb > 0;
            if (want_stats && stats_ntile != tc.n_tile) {
                if (stats_ntile >= 0) flush(stats_ntile);
                stats_ntile = tc.n_tile;
            }
#pragma unroll 1
            for (int a = 0; a < C::ACC; ++a) {
                const int64_t m = ((int64_t)tc.m_tile * CG + rank) * C::BMT + a * 128 + row;
                const bool valid = m < p.M;
                const uint32_t taddr =
                    tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((buf * C::ACC + a) * BN + cw0);
                if constexpr (FAM == kFamWgrad) {
#pragma unroll 1
                    for (int ch = 0; ch < NCH; ++ch) {
                        uint32_t v[32];
                        if (have_acc) {
                            tmem_ld_32x32b_x32(taddr + ch * 32, v);
                            tmem_ld_wait();
                        } else {
#pragma unroll
                            for (int k = 0; k < 32; ++k) v[k] = 0u;
                        }
                        const int col0 = tc.n_tile * BN + cw0 + ch * 32;
                        // D row m = (tap, c), column = output channel k; stored as [slice][k][m]:
                        // consecutive lanes hold consecutive m, so each store is one 128-byte line
                        if (valid) {
                            float* o = static_cast<float*>(p.out) + ((int64_t)tc.z * p.Ncols + col0) * p.M + m;
                            if (p.zdim == 1 && p.wg_accumulate) {
#pragma unroll
                                for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] += __uint_as_float(v[k]);
                            } else {
#pragma unroll
                                for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] = __uint_as_float(v[k]);
                            }
                        }
                    }
                } else {
                    int64_t out_row = m;
                    if (p.mode == kDgrad && p.phase_div == 2) {
                        const int64_t n = m / gPQ, rem = m - n * gPQ;
                        const int i = (int)(rem / p.gQ), j = (int)(rem - (int64_t)(rem / p.gQ) * p.gQ);
                        const int pa = tc.z >> 1, pb = tc.z & 1;
                        out_row = (n * p.out_h + 2 * i + pa) * p.out_w + 2 * j + pb;
                    }
                    const uint32_t rows_ok = __ballot_sync(0xffffffffu, valid);
#pragma unroll
                    for (int ch = 0; ch < NCH; ++ch) {
                        uint32_t v[32];
                        [[maybe_unused]] uint32_t lo[16], hi[16];
                        if (have_acc) {
                            tmem_ld_32x32b_x32(taddr + ch * 32, v);
                            if constexpr (BN > 64) {
                                if (want_stats) {
                                    tmem_ld_16x256b_x4(taddr + ch * 32, lo);
                                    tmem_ld_16x256b_x4(taddr + (16u << 16) + ch * 32, hi);
                                }
                            }
                            tmem_ld_wait_regs(v);
                            if constexpr (BN > 64) {
                                if (want_stats) {
                                    tmem_ld_wait_regs(lo);
                                    tmem_ld_wait_regs(hi);
                                }
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < 32; ++k) v[k] = 0u;
                        }
                        float back[32];
                        store_row_chunk_act(p, v, valid, out_row, tc.n_tile * BN + cw0 + ch * 32, back);
                        if constexpr (BN > 64) {  // want_stats: the forward pass, whose tiles all have K-blocks
                            if (want_stats) rs.add(ch, lo, hi, rows_ok, lane);
                        } else {
                            if (want_stats) rs.add(ch, back);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (CG == 2)
                    mbar_arrive_cluster(mapa_shared(smem_u32(&acce_bar[buf]), 0));
                else
                    mbar_arrive(&acce_bar[buf]);
            }
        }
        if (want_stats && stats_ntile >= 0) flush(stats_ntile);
        if (want_stats) {
            asm volatile("bar.sync 1, %0;" ::"r"(C::EPI * 32) : "memory");
            float* dst = p.stats + (int64_t)blockIdx.x * 2 * p.Ncols;
            for (int c = threadIdx.x; c < 2 * p.Ncols; c += C::EPI * 32)
                dst[c] = (epi_sum[c] + epi_sum[2 * p.Ncols + c]) + (epi_sum[4 * p.Ncols + c] + epi_sum[6 * p.Ncols + c]);
        }
    }
    tc_fence_before();
    __syncthreads();
    // neither CTA of a pair leaves while the other may still signal its barriers or read its TMEM
    if constexpr (CG == 2) cluster_sync_all();
    if (warp == C::MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_cg<CG>(tmem, C::TMEM_COLS);
    }
}

// ----------------------------------------------------------------------------- split-K on chip
// The 256-column pair tiles of the forward pass and the data gradient when there are too few of them
// for the GPU (the layers of a few thousand pixels): a cluster of SK CTA pairs shares one tile, pair j
// reducing K-blocks j*nkb/SK .. (j+1)*nkb/SK - 1.  When every pair's MMAs are done (cluster barrier;
// the operand rings are free), pair j owns columns j*256/SK ..: each CTA sends the other pairs'
// columns of its accumulator rows into the ring of the CTA of the same rank in those pairs
// (distributed shared memory, 16 bytes per thread and store, lanes contiguous), and after a second
// barrier adds what it received to its own columns in the pairs' order and runs the epilogue on them.
// The other pair's partial sums are fp32 as they leave TMEM, so the result is that of a different
// order of fp32 additions.
// Why: with one pair per tile a 4x4 or 3x3 map of 512 channels runs 72 K-blocks (36.9 k tensor cycles)
// on 6 to 36 of 76 pairs.  128-column tiles instead would need 1.5 times the operand bytes per MMA.
// Channel sums: the CTAs of a row block write disjoint columns of one partial row (2 * m_tiles rows).
// The weight gradient's pair tiles share their K range the same way where that saves slices of fp32 partial
// sums (p.zdim of them are left for wgrad_reduce_kernel; none when it is 1): 7x7x512,
// batch 512 91.6 -> 85.7 us and 128 32.1 -> 27.1, 3x3x512, batch 512 26.7 -> 22.0, 12x12 128 -> 256 stride 2,
// batch 512 25.7 -> 20.8, a 14x14 projection 256 -> 512, batch 128 15.9 -> 13.0 (with the reduce).
template <int BN, int FAM, int SK>
struct SplitCfg {
    using C = Cfg<BN, FAM, 2>;
    static_assert(C::ACC == 1 && BN / SK >= 32, "one accumulator, whole chunks");
    // The weight gradient's K ranges are longer than the slices they replace, and the tensor core's sums lose with
    // their length (it rounds towards zero): each half of the range has an accumulator of its own, added in
    // fp32.  4x4x256, batch 256: error of dw against 64 bits 8.4e-7 with one, 4.0e-7 with two, 13.8 us both.
    static constexpr int ACCS = FAM == kFamWgrad ? 2 : 1;
    static constexpr uint32_t TMEM_COLS = ACCS * BN;
    static constexpr int EPI = 8, MMA_WARP = EPI + kProducers, THREADS = 32 * (MMA_WARP + 1);
    static constexpr int W = BN / SK;              // columns a CTA finishes
    static constexpr int SLOT = 128 * W * 4;        // one received part: [W / 4][128 rows] float4
    static constexpr int CW = W > 32 ? W / 2 : 32;  // columns an epilogue warp finishes (of W = 32: one warp per quarter)
    static constexpr int EPI_TILE = FAM == kFamFwd ? 8 * 32 * 33 * 4 : 0;  // transposes of the channel sums
    static constexpr int EPI_SUM = 4 * 2 * W * 4;   // channel sums per lane quarter
    static constexpr int SMEM = C::RING + EPI_SUM + 1024;
    static_assert((SK - 1) * SLOT + EPI_TILE <= C::RING, "received parts and transposes fit in the ring");
};

template <int BN, int FAM, int SK>
__global__ void __launch_bounds__(SplitCfg<BN, FAM, SK>::THREADS, 1)
    conv_splitk_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
                       const ConvParams p)
{
    using S = SplitCfg<BN, FAM, SK>;
    using C = typename S::C;
    constexpr int STAGES = C::STAGES, W = S::W;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], accf_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    const int crank = (int)cluster_ctarank(), rank = crank & 1, split = crank >> 1;
    const uint32_t leader = (uint32_t)(crank & ~1);  // the CTA of this pair that issues its MMAs
    const int t = blockIdx.x / (2 * SK);
    const TileCoord tc = decode_tile(p, t, gridDim.x);
    int k0 = 0, nkb = 0;  // this pair's K-blocks
    if constexpr (FAM == kFamWgrad) {
        k0 = (tc.z * SK + split) * p.kb_per_split;
        nkb = max(0, min(p.num_kb, k0 + p.kb_per_split) - k0);
    } else {
        int first = 0, all = 0;
        kb_range(p, tc.z, first, all);
        k0 = all * split / SK;
        nkb = all * (split + 1) / SK - k0;
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&accf_bar, 1);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    if (warp >= S::EPI && warp < S::MMA_WARP && lane == 0) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        if (p.proj_kb) {
            tma_prefetch_desc(&tmA2);
            tma_prefetch_desc(&tmB2);
        }
    }
    if (warp == S::MMA_WARP) {
        tmem_alloc_cg<2>(&tmem_slot, S::TMEM_COLS);
        tmem_relinquish_cg<2>();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // every CTA's barriers initialised, TMEM allocated
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;
    const int64_t gPQ = (int64_t)p.gP * p.gQ;
    const int nkb_first = S::ACCS == 2 ? (nkb + 1) / 2 : nkb;  // K-blocks of the first accumulator

    if (warp >= S::EPI && warp < S::MMA_WARP) {
        // ------------------------------------------------------------------ TMA producers
        const int prod = warp - S::EPI;
        int tn = 0, tp = 0, tq = 0;
        if constexpr (FAM == kFamFwd) {
            const int64_t m0 = ((int64_t)tc.m_tile * 2 + rank) * 128;
            tn = (int)(m0 / gPQ);
            const int64_t rem = m0 - (int64_t)tn * gPQ;
            tp = (int)(rem / p.gQ);
            tq = (int)(rem - (int64_t)tp * p.gQ);
        }
        bool failed = false;
        int last_it = -1;
        for (int k = prod; k < nkb; k += kProducers) {
            if (p.test_stall && blockIdx.x == 0 && k == 0) continue;  // stage 0 never fills (bounded-wait test)
            const int s = k % STAGES;
            const uint32_t ok = mbar_wait_warp(&empty_bar[s], ((k / STAGES) & 1) ^ 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                failed = true;
                break;
            }
            uint8_t* sa = sgen + s * C::STAGE_BYTES;
            if (rank == 0) mbar_arrive_expect_tx_elect(&full_bar[s], (uint32_t)(2 * C::STAGE_BYTES));
            load_kblock<BN, FAM, 2>(p, &tmA, &tmB, &tmA2, &tmB2, sa, sa + C::A_BYTES,
                                        mapa_shared(smem_u32(&full_bar[s]), leader), tc, k0 + k, tn, tp, tq, rank);
            last_it = k;
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            if (rank == 0) {
                // let copies this producer issued land before the shared memory is used for anything else
                for (int i = last_it; i >= 0 && i > last_it - STAGES * kProducers; i -= kProducers)
                    (void)mbar_drain_warp(&full_bar[i % STAGES], (i / STAGES) & 1);
            } else {
                // rank 1's copies complete on rank 0's barriers: give them a fixed time instead
                const uint64_t t0 = globaltimer();
                while (globaltimer() - t0 < 1000000ull) {
                }
            }
        }
    } else if (warp == S::MMA_WARP) {
        // ------------------------------------------------------------------ MMA issuer (rank 0 of each pair)
        if (rank == 0) {
            // operand layouts as in conv_igemm_kernel
            const bool wg = FAM == kFamWgrad, fwd = p.mode == kFwd;
            const uint32_t idesc = idesc_act(BM * 2, BN, wg ? 1u : 0u, fwd ? 0u : 1u);
            const uint16_t both = (uint16_t)(3u << leader);
            const uint64_t dA = smem_desc(0, wg ? 16384 : 16, 1024, kSwizzle128B);
            const uint64_t dB = smem_desc(0, wg ? 16384 : fwd ? 16 : 8192, 1024, kSwizzle128B);
            const int a_step16 = wg ? 2048 / 16 : 2, b_step16 = fwd ? 2 : 2048 / 16;
            bool failed = false;
            if (nkb > 0) {
                const uint32_t ok = mbar_wait_warp(&full_bar[0], 0, &abort_flag);
                failed = __any_sync(0xffffffffu, ok == 0u);
            }
            for (int k = 0; k < nkb && !failed; ++k) {
                tc_fence_after();
                const int s = k % STAGES;
                const uint32_t sa = sbase + s * C::STAGE_BYTES, sb = sa + C::A_BYTES;
                const uint64_t ad0 = dA | (uint64_t)((sa >> 4) & 0x3FFFu), bd0 = dB | (uint64_t)((sb >> 4) & 0x3FFFu);
                const uint32_t d = tmem + (k >= nkb_first ? (uint32_t)BN : 0u);
                const bool held = k != 0 && k != nkb_first;  // the accumulator holds a K-block already
#pragma unroll
                for (int j = 0; j < C::KSTEPS; ++j) {
                    if (j == C::KSTEPS - 1 && k + 1 < nkb) {  // the next stage's wait while MMAs are queued
                        const uint32_t ok =
                            mbar_wait_warp(&full_bar[(k + 1) % STAGES], ((k + 1) / STAGES) & 1, &abort_flag);
                        failed = __any_sync(0xffffffffu, ok == 0u);
                    }
                    mma_act_elect_cg<2>(d, ad0 + (uint64_t)(j * a_step16), bd0 + (uint64_t)(j * b_step16), idesc,
                                        (held || j > 0) ? 1u : 0u);
                }
                mma_commit_elect_cg<2>(&empty_bar[s], both);
            }
            mma_commit_elect_cg<2>(&accf_bar, both);  // arrives when this pair's MMAs have completed
            if (failed && lane == 0) report_timeout(&abort_flag);
            mma_commit_elect_cg<2>(&drain_bar, (uint16_t)(1u << leader));
            (void)mbar_drain_warp(&drain_bar, 0);
        }
    } else {
        const uint32_t ok = mbar_wait_warp(&accf_bar, 0, &abort_flag);
        if (__any_sync(0xffffffffu, ok == 0u) && lane == 0) report_timeout(&abort_flag);
        tc_fence_after();
    }
    __syncwarp();
    cluster_sync_all();  // every pair's MMAs are done: the rings may be overwritten

    const int quarter = warp & 3, half = warp >> 2;  // epilogue warps (0-7): TMEM lanes 32*quarter..
    const int row = quarter * 32 + lane;             // row within the 128-row accumulator
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
    constexpr int CW = S::CW, NCH = CW / 32;
    const bool finishes = warp < S::EPI && half * CW < W;
    auto load_acc = [&](uint32_t col, uint32_t(&v)[32]) {  // 32 columns of the accumulator, or of both
        tmem_ld_32x32b_x32(taddr + col, v);
        if (S::ACCS == 2 && nkb > nkb_first) {
            uint32_t u[32];
            tmem_ld_32x32b_x32(taddr + BN + col, u);
            tmem_ld_wait_regs(v);
            tmem_ld_wait_regs(u);
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] = __float_as_uint(__uint_as_float(v[k]) + __uint_as_float(u[k]));
        } else {
            tmem_ld_wait_regs(v);
        }
    };
    uint32_t own[NCH][32];  // this warp's part of the CTA's own columns
    if (warp < S::EPI) {
        // the other pairs' chunks of 32 columns, the two warps of a quarter taking alternate ones
#pragma unroll 1
        for (int e = half; e < (SK - 1) * (W / 32); e += 2) {
            const int to = (split + 1 + e / (W / 32)) % SK;   // pair that finishes these columns
            const int ch = e % (W / 32);
            const int slot = split < to ? split : split - 1;  // its parts are kept in the pairs' order
            const uint32_t dst = mapa_shared(sbase, (uint32_t)(2 * to + rank)) + (uint32_t)(slot * S::SLOT + row * 16);
            uint32_t v[32];
            if (nkb > 0) {
                load_acc((uint32_t)(to * W + ch * 32), v);
            } else {
#pragma unroll
                for (int k = 0; k < 32; ++k) v[k] = 0u;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                st_cluster_v4(dst + (uint32_t)((ch * 8 + k) * 2048), v[4 * k], v[4 * k + 1], v[4 * k + 2],
                              v[4 * k + 3]);
        }
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            if (nkb > 0 && finishes) {
                load_acc((uint32_t)(split * W + half * CW + ch * 32), own[ch]);
            } else {
#pragma unroll
                for (int k = 0; k < 32; ++k) own[ch][k] = 0u;
            }
        }
        tc_fence_before();
    }
    __syncwarp();
    cluster_sync_all();  // the parts have arrived, and every accumulator has been read
    if (warp == S::MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_cg<2>(tmem, S::TMEM_COLS);
    }

    if (warp < S::EPI) {
        // ------------------------------------------------------------------ epilogue of this CTA's columns
        float* sums = reinterpret_cast<float*>(sgen + C::RING);
        const bool want_stats = FAM == kFamFwd && p.mode == kFwd && p.stats != nullptr;
        const int64_t m = ((int64_t)tc.m_tile * 2 + rank) * 128 + row;
        const bool valid = m < p.M;
        int64_t out_row = m;
        if (p.mode == kDgrad && p.phase_div == 2) {
            const int64_t n = m / gPQ, rem = m - n * gPQ;
            const int i = (int)(rem / p.gQ), j = (int)(rem - (int64_t)(rem / p.gQ) * p.gQ);
            out_row = (n * p.out_h + 2 * i + (tc.z >> 1)) * p.out_w + 2 * j + (tc.z & 1);
        }
        if (finishes) {
            RowStats<CW> rs;
            rs.zero();
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) {
                uint32_t(&v)[32] = own[ch];
                const float4* src = reinterpret_cast<const float4*>(sgen + (half * NCH + ch) * 8 * 2048 + row * 16);
#pragma unroll
                for (int q = 0; q < SK - 1; ++q)
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 f = src[q * (S::SLOT / 16) + k * 128];
                        v[4 * k] = __float_as_uint(__uint_as_float(v[4 * k]) + f.x);
                        v[4 * k + 1] = __float_as_uint(__uint_as_float(v[4 * k + 1]) + f.y);
                        v[4 * k + 2] = __float_as_uint(__uint_as_float(v[4 * k + 2]) + f.z);
                        v[4 * k + 3] = __float_as_uint(__uint_as_float(v[4 * k + 3]) + f.w);
                    }
                const int col0 = tc.n_tile * BN + split * W + half * CW + ch * 32;
                if constexpr (FAM == kFamWgrad) {
                    // [slice][k][m]: consecutive lanes hold consecutive m, one 128-byte line per store
                    float* o = static_cast<float*>(p.out) + ((int64_t)tc.z * p.Ncols + col0) * p.M + m;
                    if (valid && p.zdim == 1 && p.wg_accumulate) {
#pragma unroll
                        for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] += __uint_as_float(v[k]);
                    } else if (valid) {
#pragma unroll
                        for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] = __uint_as_float(v[k]);
                    }
                } else {
                    float back[32];
                    store_row_chunk_act(p, v, valid, out_row, col0, back);
                    if (want_stats) rs.add(ch, back);
                }
            }
            if (want_stats) {
                float* st_tile = reinterpret_cast<float*>(sgen + (SK - 1) * S::SLOT) + warp * 32 * 33;
                float* wsum = sums + quarter * 2 * W;
                for (int c = lane; c < 2 * CW; c += 32) wsum[(c / CW) * W + half * CW + c % CW] = 0.f;
                __syncwarp();
                rs.flush(st_tile, wsum, W, half * CW, lane);
            }
        }
        if (want_stats) {
            asm volatile("bar.sync 1, 256;" ::: "memory");
            float* dst = p.stats + (int64_t)(tc.m_tile * 2 + rank) * 2 * p.Ncols + tc.n_tile * BN + split * W;
            for (int c = threadIdx.x; c < 2 * W; c += 256)
                dst[(c / W) * p.Ncols + c % W] = (sums[c] + sums[2 * W + c]) + (sums[4 * W + c] + sums[6 * W + c]);
        }
    }
}

// ----------------------------------------------------------------------------- window kernel
// 3x3, stride-1, pad-1 correlation (the forward pass, and the data gradient
// with the taps flipped) without im2col.  Position (h, w) of image n of the
// zero-padded input is row g = n*Hp + h of a column of padded rows, and
// padded position L = g*Wp + w.  Output (h, w) of image n is computed at
// L = (n*Hp + h)*Wp + w, and its tap (r, s) reads padded position L + r*Wp + s.
// So a tile of 256 consecutive L needs one strip of padded rows (TMA loads
// one padded row per copy: the box starts at w = -1 and the zero fill makes
// the padding), and each of the nine taps is the same strip addressed by a
// descriptor that starts r*Wp + s rows later.  The 128-byte swizzle of both
// TMA and the MMA operand fetch is a function of the absolute shared-memory
// address, so a start at any 128-byte row reads the rows that TMA wrote.  Rows
// with h >= H or w >= W are computed and not stored (the padding's share of
// the work: 7% at 56x56, 13% at 28x28).
// Warp roles (WinCfg): a producer of strips (two buffers), a producer of weights (all
// nine taps once per CTA when they fit, RES; else a ring of per-tap tiles), the MMA
// issuer, and four or eight warps that drain TMEM as in conv_igemm_kernel.
constexpr int kWinACC = 2;               // 128-row accumulators per tile
constexpr int kWinBMT = 128 * kWinACC;   // padded positions per tile
constexpr int kWinBStages = 4;           // weight-tile ring depth when not resident
constexpr int kWinThreads = 224;         // weight gradients: 4 epilogue warps, 2 producers, MMA

// Warp roles of conv_win_kernel: EPI epilogue warps (0 .. EPI-1), then the strip
// producer, the weight producer and the MMA issuer.  128-column tiles drain with eight epilogue
// warps, two per TMEM lane quarter; 64-column ones (the stem) with four: eight there, and stores staged
// in shared memory so that each instruction writes whole lines, both measured slower.
template <int BN>
struct WinCfg {
    static constexpr int B_TILE = BN * 64 * 2;  // one tap x one 64-channel block of weights
    static constexpr int NB = BN == 64 ? 4 : 2;  // accumulator buffers (tiles in flight)
    static constexpr uint32_t TMEM_COLS = NB * kWinACC * BN;
    static constexpr int EPI = BN == 128 ? 8 : 4;  // epilogue warps
    static constexpr int CW = BN * 4 / EPI;      // columns one epilogue warp drains
    static constexpr int W_STRIP = EPI, W_WEIGHT = EPI + 1, W_MMA = EPI + 2;
    static constexpr int THREADS = 32 * (EPI + 3);
};

// One tap x 64-channel block of weights: K-major [BN out][64 in] for the forward
// pass, MN-major [64 k][BN c] blocks of 64 for the data gradient (flipped tap).
// CG = 2: this CTA's half of the BN columns (rank r: columns r*BN/2 ..), completing
// on the barrier at shared::cluster address bar (the leader's).
template <int BN, bool DG, int CG>
__device__ __forceinline__ void win_load_wtile(const ConvParams& p, const CUtensorMap* tmB, uint8_t* dst, uint32_t bar,
                                               int tap, int cb, int n_tile, int rank)
{
    if constexpr (DG) {
        const int wtap = p.win_R * p.win_S - 1 - tap;  // flipped filter
#pragma unroll
        for (int j = 0; j < BN / 64 / CG; ++j)
            tma_load_3d_cg<CG>(dst + j * 8192, tmB, bar, n_tile * BN + rank * (BN / CG) + 64 * j, wtap, cb * 64);
    } else {
        tma_load_2d_cg<CG>(dst, tmB, bar, tap * p.Cin + cb * 64, n_tile * BN + rank * (BN / CG));
    }
}

// CG = 2 (a cluster of two CTAs, tcgen05 .cta_group::2): CTA rank r computes tile
// 2u + r of pair unit u.  Rank 0 issues M = 256 MMAs whose A rows 0-127 come from
// its strip and rows 128-255 from rank 1's, at the same shared-memory address, and
// whose B columns are split between the two CTAs' halves of the weights, so each SM
// reads half of B per MMA.  The two tiles start at different offsets within a
// padded row (off0), so rank 1 places its strip (off0 of rank 0 - off0 of rank 1)
// rows away from rank 0's (inside a margin of one padded row on either side): the
// descriptors rank 0 builds from its own off0 then read rank 1's tile at the same
// rows.  Rank 0 owns the strip-full, weight-full and accumulator-empty barriers;
// both CTAs' copies complete on rank 0's full barriers, rank 0's commits arrive on
// both CTAs' empty and accumulator-full barriers, and both CTAs' epilogues arrive on
// rank 0's accumulator-empty barrier.  A pair unit past the last tile loads zeros
// (images past the batch) and stores nothing.
template <int BN, bool DG, bool RES, int CG>
__global__ void __launch_bounds__(WinCfg<BN>::THREADS, 1)
    conv_win_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const ConvParams p)
{
    using C = WinCfg<BN>;
    static_assert(CG == 1 || BN == 128 || !DG, "data-gradient pairs split the weights in 64-column halves");
    constexpr int BT = C::B_TILE / CG;  // this CTA's bytes of one tap x 64-channel block of weights
    constexpr uint16_t kAll = CG == 2 ? 3 : 1;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t sfull[2], sempty[2], bfull[kWinBStages], bempty[kWinBStages], accf_bar[4],
        acce_bar[4], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    const int rank = CG == 2 ? (int)cluster_ctarank() : 0;
    const int unit0 = blockIdx.x / CG, nunits = gridDim.x / CG;
    const int total_units = (p.total_tiles + CG - 1) / CG;
    const int CB = p.cblocks;
    const int ntaps = p.win_R * p.win_S;
    const int b_bytes = RES ? ntaps * CB * BT : kWinBStages * BT;
    const int strip_stride = p.win_strip_bytes + 2 * p.win_margin;
    uint8_t* strip = sgen + b_bytes + p.win_margin;  // stage s at strip + s * strip_stride
    // per-warp statistics transposes reuse the strip buffers once the last tile's MMAs are done
    float* epi_tile = reinterpret_cast<float*>(sgen + b_bytes);
    float* epi_sum = reinterpret_cast<float*>(sgen + b_bytes + 2 * strip_stride);

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sfull[i], 1);
            mbar_init(&sempty[i], 1);
        }
        for (int i = 0; i < C::NB; ++i) {
            mbar_init(&accf_bar[i], 1);
            mbar_init(&acce_bar[i], C::EPI * CG);  // one arrival per epilogue warp of the pair
        }
        for (int i = 0; i < kWinBStages; ++i) {
            mbar_init(&bfull[i], 1);
            mbar_init(&bempty[i], 1);
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    const bool want_stats = p.mode == kFwd && p.stats != nullptr;
    if (want_stats)
        for (int i = threadIdx.x; i < C::EPI * 2 * p.Ncols; i += blockDim.x) epi_sum[i] = 0.f;
    if ((warp == C::W_STRIP || warp == C::W_WEIGHT) && lane == 0) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == C::W_MMA) {
        tmem_alloc_cg<CG>(&tmem_slot, C::TMEM_COLS);
        tmem_relinquish_cg<CG>();
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) cluster_sync_all();  // both CTAs' barriers initialised, TMEM allocated
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;
    const int Wp = p.win_Wp;

    if (warp == C::W_STRIP) {
        // ------------------------------------------------------------------ strip producer
        int it = 0;
        bool failed = false;
        const uint32_t strip_tx = (uint32_t)(p.win_srows * Wp * 128);
        for (int t = unit0; t < total_units; t += nunits) {
            const int m_tile = t * CG + rank;
            const int L0 = m_tile * p.win_tile;
            const int g0 = L0 / Wp, n0 = g0 / p.win_Hp, hp0 = g0 - n0 * p.win_Hp;
            // rank 1: rows between its strip and rank 0's, so that both tiles sit at rank 0's offsets
            const int shift = (CG == 2 && rank == 1) ? ((L0 - p.win_tile) % Wp) - (L0 % Wp) : 0;
            for (int cb = 0; cb < CB; ++cb, ++it) {
                const int s = it & 1;
                const uint32_t ok = mbar_wait_warp(&sempty[s], ((it >> 1) & 1) ^ 1, &abort_flag);
                if (__any_sync(0xffffffffu, ok == 0u)) {
                    failed = true;
                    break;
                }
                uint8_t* dst = strip + s * strip_stride + shift * 128;
                uint32_t fb = smem_u32(&sfull[s]);
                if (CG == 1 || rank == 0) mbar_arrive_expect_tx_elect(&sfull[s], (uint32_t)CG * strip_tx);
                if (CG == 2) fb = mapa_shared(fb, 0);
                int n = n0, hp = hp0;
                for (int r = 0; r < p.win_srows; ++r) {
                    // padded row hp of image n = input row hp - ph from column -pw (padding rows and
                    // columns, and images past the batch, are outside the tensor and arrive as zeros)
                    tma_load_4d_cg<CG>(dst + r * Wp * 128, &tmA, fb, cb * 64, -p.win_pw, hp - p.win_ph, n);
                    if (++hp == p.win_Hp) {
                        hp = 0;
                        ++n;
                    }
                }
            }
            if (failed) break;
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            if (CG == 1 || rank == 0) {
                for (int i = it - 1; i >= 0 && i >= it - 2; --i) (void)mbar_drain_warp(&sfull[i & 1], (i >> 1) & 1);
            } else {
                // rank 1's copies complete on rank 0's barriers: give them a fixed time instead
                const uint64_t t0 = globaltimer();
                while (globaltimer() - t0 < 1000000ull) {
                }
            }
        }
    } else if (warp == C::W_WEIGHT) {
        // ------------------------------------------------------------------ weight producer
        if (RES) {
            uint32_t fb = smem_u32(&bfull[0]);
            if (CG == 1 || rank == 0) mbar_arrive_expect_tx_elect(&bfull[0], (uint32_t)(CG * ntaps * CB * BT));
            if (CG == 2) fb = mapa_shared(fb, 0);
            for (int tap = 0; tap < ntaps; ++tap)
                for (int cb = 0; cb < CB; ++cb)
                    win_load_wtile<BN, DG, CG>(p, &tmB, sgen + (tap * CB + cb) * BT, fb, tap, cb, 0, rank);
            if (CG == 1 || rank == 0) (void)mbar_drain_warp(&bfull[0], 0);
        } else {
            int bt = 0;
            bool failed = false;
            for (int t = unit0; t < total_units && !failed; t += nunits)
                for (int cb = 0; cb < CB && !failed; ++cb)
                    for (int tap = 0; tap < ntaps; ++tap, ++bt) {
                        const int s = bt % kWinBStages;
                        const uint32_t ok =
                            mbar_wait_warp(&bempty[s], ((bt / kWinBStages) & 1) ^ 1, &abort_flag);
                        if (__any_sync(0xffffffffu, ok == 0u)) {
                            failed = true;
                            break;
                        }
                        uint32_t fb = smem_u32(&bfull[s]);
                        if (CG == 1 || rank == 0) mbar_arrive_expect_tx_elect(&bfull[s], (uint32_t)(CG * BT));
                        if (CG == 2) fb = mapa_shared(fb, 0);
                        win_load_wtile<BN, DG, CG>(p, &tmB, sgen + s * BT, fb, tap, cb, 0, rank);
                    }
            if (failed) {
                if (lane == 0) report_timeout(&abort_flag);
                if (CG == 1 || rank == 0) {
                    for (int i = bt - 1; i >= 0 && i >= bt - kWinBStages; --i)
                        (void)mbar_drain_warp(&bfull[i % kWinBStages], (i / kWinBStages) & 1);
                } else {
                    const uint64_t t0 = globaltimer();
                    while (globaltimer() - t0 < 1000000ull) {
                    }
                }
            }
        }
    } else if (warp == C::W_MMA) {
        // ------------------------------------------------------------------ MMA issuer (rank 0 of a pair)
        const uint32_t idesc = idesc_act(BM * CG, BN, 0u, DG ? 1u : 0u);
        int it = 0, bt = 0, lt = 0;
        bool failed = false;
        if (RES && (CG == 1 || rank == 0)) {
            const uint32_t ok = mbar_wait_warp(&bfull[0], 0, &abort_flag);
            failed = __any_sync(0xffffffffu, ok == 0u);
        }
        for (int t = unit0; t < total_units && (CG == 1 || rank == 0) && !failed; t += nunits, ++lt) {
            const int buf = lt % C::NB;
            const uint32_t ok = mbar_wait_warp(&acce_bar[buf], ((lt / C::NB) & 1) ^ 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                failed = true;
                break;
            }
            tc_fence_after();
            const int L0 = t * CG * p.win_tile;  // this CTA's (rank 0's) tile
            const int off0 = L0 - (L0 / Wp) * Wp;  // tile start within the strip's first row
            const uint32_t d = tmem + (uint32_t)(buf * kWinACC * BN);
            for (int cb = 0; cb < CB && !failed; ++cb, ++it) {
                const int s = it & 1;
                const uint32_t oks = mbar_wait_warp(&sfull[s], (it >> 1) & 1, &abort_flag);
                if (__any_sync(0xffffffffu, oks == 0u)) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = smem_u32(strip + s * strip_stride);
                int r = 0, sx = 0;  // (tap / S, tap % S), stepped without divisions
#pragma unroll 1
                for (int tap = 0; tap < ntaps; ++tap) {
                    uint32_t sb;
                    int bs = 0;
                    if (RES) {
                        sb = sbase + (uint32_t)((tap * CB + cb) * BT);
                    } else {
                        bs = bt % kWinBStages;
                        const uint32_t okb = mbar_wait_warp(&bfull[bs], (bt / kWinBStages) & 1, &abort_flag);
                        if (__any_sync(0xffffffffu, okb == 0u)) {
                            failed = true;
                            break;
                        }
                        tc_fence_after();
                        sb = sbase + (uint32_t)(bs * BT);
                    }
                    const uint32_t a0 = sa + (uint32_t)((off0 + r * Wp + sx) * 128);
                    // K-step j of accumulator a: A rows a*128.. of the shifted strip, 32 bytes per K-step;
                    // B K-major (32 bytes per K-step) or, for the data gradient, MN-major (2 KB per K-step)
                    static_assert(kWinACC == 2, "two accumulators per MMA group");
                    const uint64_t ad = smem_desc(a0, 16, 1024, kSwizzle128B);
                    const uint64_t bd = DG ? smem_desc(sb, 8192, 1024, kSwizzle128B) : smem_desc(sb, 16, 1024, kSwizzle128B);
                    mma_act_x8_elect_cg<CG>(d, d + BN, ad, (128 * 128) >> 4, 32 >> 4, bd, DG ? (2048 >> 4) : (32 >> 4),
                                             idesc, (cb > 0 || tap > 0) ? 1u : 0u);
                    if (!RES) {
                        mma_commit_elect_cg<CG>(&bempty[bs], kAll);
                        ++bt;
                    }
                    if (++sx == p.win_S) {
                        sx = 0;
                        ++r;
                    }
                }
                mma_commit_elect_cg<CG>(&sempty[s], kAll);
            }
            mma_commit_elect_cg<CG>(&accf_bar[buf], kAll);  // arrives when this unit's MMAs have completed
        }
        if (CG == 1 || rank == 0) {
            if (failed && lane == 0) report_timeout(&abort_flag);
            mma_commit_elect_cg<CG>(&drain_bar, 1);
            (void)mbar_drain_warp(&drain_bar, 0);
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 0 .. EPI-1)
        constexpr int CW = C::CW;
        const int quarter = warp & 3, col0 = (warp >> 2) * CW;  // TMEM lanes 32*quarter.., columns col0..
        float* st_tile = epi_tile + warp * 32 * 33;
        float* wsum = epi_sum + warp * 2 * p.Ncols;
        TileStats<BN> rs;
        rs.zero();
        const int img = p.win_Hp * Wp;
        int lt = 0;
        for (int t = unit0; t < total_units; t += nunits, ++lt) {
            const int m_tile = t * CG + rank;
            const int buf = lt % C::NB;
            const uint32_t ok = mbar_wait_warp(&accf_bar[buf], (lt / C::NB) & 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                if (lane == 0) report_timeout(&abort_flag);
                break;
            }
            tc_fence_after();
            const int row = quarter * 32 + lane;
            bool valid[kWinACC];
            int64_t out_row[kWinACC];
#pragma unroll
            for (int a = 0; a < kWinACC; ++a) {
                const int L = m_tile * p.win_tile + a * 128 + row;
                const int n = L / img, rem = L - n * img;
                const int hp = rem / Wp, wp = rem - hp * Wp;
                // rows past the tile belong to the next tile (row-aligned tiles are shorter than 256)
                valid[a] = m_tile < p.total_tiles && a * 128 + row < p.win_tile && n < p.gN && hp < p.win_P &&
                           wp < p.win_Q;
                out_row[a] = ((int64_t)n * p.win_P + hp) * p.win_Q + wp;
            }
            // chunks c = (accumulator, 32 of this warp's columns)
            const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kWinACC * BN + col0);
            constexpr int NCH = CW / 32, NC = kWinACC * NCH;
            // the next chunk's TMEM load in flight while this one is converted and stored
            uint32_t va[32], vb[32];
            tmem_ld_32x32b_x32(taddr, va);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                uint32_t(&cur)[32] = (c & 1) ? vb : va;
                uint32_t(&nxt)[32] = (c & 1) ? va : vb;
                tmem_ld_wait_regs(cur);
                const int a = c / NCH, ch = c % NCH;
                if (c + 1 < NC)
                    tmem_ld_32x32b_x32(taddr + (uint32_t)(((c + 1) / NCH) * BN + ((c + 1) % NCH) * 32), nxt);
                float back[32];
                if constexpr (BN > 64) {
                    uint32_t lo[16], hi[16];
                    if (want_stats) {
                        const uint32_t ta = taddr + (uint32_t)(a * BN + ch * 32);
                        tmem_ld_16x256b_x4(ta, lo);
                        tmem_ld_16x256b_x4(ta + (16u << 16), hi);
                    }
                    store_row_chunk_act(p, cur, valid[a], out_row[a], col0 + ch * 32, back);
                    if (want_stats) {
                        const uint32_t rows_ok = __ballot_sync(0xffffffffu, valid[a]);
                        tmem_ld_wait_regs(lo);
                        tmem_ld_wait_regs(hi);
                        rs.add(ch, lo, hi, rows_ok, lane);
                    }
                } else {
                    store_row_chunk_act(p, cur, valid[a], out_row[a], col0 + ch * 32, back);
                    if (want_stats) rs.add(ch, back);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (CG == 2)
                    mbar_arrive_cluster(mapa_shared(smem_u32(&acce_bar[buf]), 0));
                else
                    mbar_arrive(&acce_bar[buf]);
            }
        }
        if (want_stats) {
            if constexpr (BN > 64)
                rs.flush(wsum, p.Ncols, col0, lane);  // the window kernel has one column tile
            else
                rs.flush(st_tile, wsum, p.Ncols, col0, lane);
            asm volatile("bar.sync 1, %0;" ::"r"(C::EPI * 32) : "memory");
            float* dst = p.stats + (int64_t)blockIdx.x * 2 * p.Ncols;
            const int nc = 2 * p.Ncols;
            // warps 4g..4g+3 hold column group g; the other groups' rows are zero
            for (int c = threadIdx.x; c < nc; c += C::EPI * 32) {
                float v = (epi_sum[c] + epi_sum[nc + c]) + (epi_sum[2 * nc + c] + epi_sum[3 * nc + c]);
                if constexpr (C::EPI == 8)
                    v += (epi_sum[4 * nc + c] + epi_sum[5 * nc + c]) + (epi_sum[6 * nc + c] + epi_sum[7 * nc + c]);
                dst[c] = v;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    // neither CTA of a pair leaves while the other may still signal its barriers or read its TMEM
    if constexpr (CG == 2) cluster_sync_all();
    if (warp == C::W_MMA) {
        tc_fence_after();
        tmem_dealloc_cg<CG>(tmem, C::TMEM_COLS);
    }
}

// ----------------------------------------------------------------------------- window kernel, pixel pairs
// 3x3 stride-1 pad-1 correlation of 64 to 64 channels (forward, or the data gradient with the taps
// flipped) with an even row width.  An accumulator row is a pair of neighbouring pixels (2j, 2j + 1) and
// its 128 columns are both pixels' 64 outputs, which are contiguous in memory.  The strip holds the
// even and the odd pixels of a padded row apart (E, O: 64-channel strips of W/2 + 1 entries, the first a
// zero that also pads the row before), so that the four input pixels a pair's filter row reads are
//     O[j-1]: w0 to the even output          (N = 64)
//     E[j]:   w1 to the even, w0 to the odd  (N = 128)
//     O[j]:   w2 to the even, w1 to the odd  (N = 128)
//     E[j+1]: w2 to the odd                  (N = 64)
// With the resident weight tiles of a filter row stored in the order w2, w1, w0 every B operand is one run
// of them, and in this order every output adds its taps as conv_win_kernel does (the same bits).  256 pixels take 24 MMAs of 64 columns and 24 of 128 instead of 72 of 64, which are bound by
// their operand reads and issue (54 against ~70 cycles each): forward at 56x56, batch 512 112 -> 91 us,
// data gradient 110 -> 89; 72x72, batch 185 79 -> 57 and 77 -> 55; 24x24, batch 512 27.9 -> 23.2 and 26.5 -> 21.5;
// 32x32, batch 64 11.2 -> 10.1 and 10.3 -> 8.8.
// CG = 2 (forward only, selected by DBL_CONV_CTA_PAIRS=2): two CTAs, each with its own tile, as M = 256 MMAs;
// each holds half of every B operand, one pixel's tap for N = 128 and 32 outputs for N = 64, and rank 1
// shifts its strips as in conv_win_kernel.
// Warp roles as in conv_win_kernel: warps 0-3 drain TMEM, 4 loads strips, 5 the weights, 6 issues MMAs.
constexpr int kPairNB = 4;  // accumulator buffers of 128 columns

template <bool DG, int CG>
__global__ void __launch_bounds__(kWinThreads, 1)
    conv_winpair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmB32, const ConvParams p)
{
    static_assert(CG == 1 || !DG, "a 32-column half of an MN-major operand has no layout");
    constexpr int BT = 64 * 64 * 2;  // one tap of weights
    // Resident weights.  CG = 1: tap (r, s) at slot 3r + 2 - s.  CG = 2, per filter row r: this rank's tap of
    // the two N = 128 operands, then its 32 outputs of w0 and of w2; behind them 32 outputs of (0, w1).
    constexpr int kWeights = CG == 1 ? 9 * BT : 9 * BT + BT / 2;
    constexpr uint16_t kAll = CG == 2 ? 3 : 1;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t sfull[2], sempty[2], wfull, accf_bar[kPairNB], acce_bar[kPairNB], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    const int rank = CG == 2 ? (int)cluster_ctarank() : 0;
    const int unit0 = blockIdx.x / CG, nunits = gridDim.x / CG, total_units = (p.total_tiles + CG - 1) / CG;
    const int pitch = p.win_Wp, half_bytes = p.win_strip_bytes;  // one parity's strip, with rank 1's shift
    uint8_t* strip = sgen + (CG == 1 ? kWeights : (kWeights + 1023) / 1024 * 1024);  // stage s, parity e: + (2s + e) * half_bytes
    float* epi_tile = reinterpret_cast<float*>(strip);  // once the last tile's MMAs are done
    float* epi_sum = reinterpret_cast<float*>(strip + 4 * half_bytes);
    // entry of a strip buffer at which rank 0's strip starts: room for rank 1's shift of -(128 % pitch)
    const int first = CG == 2 ? p.win_margin : 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sfull[i], 1);
            mbar_init(&sempty[i], 1);
        }
        mbar_init(&wfull, 1);
        for (int i = 0; i < kPairNB; ++i) {
            mbar_init(&accf_bar[i], 1);
            mbar_init(&acce_bar[i], 4 * CG);  // one arrival per epilogue warp
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    const bool want_stats = !DG && p.stats != nullptr;
    if (want_stats)
        for (int i = threadIdx.x; i < 4 * 2 * 64; i += blockDim.x) epi_sum[i] = 0.f;
    if ((warp == 4 || warp == 5) && lane == 0) tma_prefetch_desc(warp == 4 ? &tmA : &tmB);
    if (warp == 6) {
        tmem_alloc_cg<CG>(&tmem_slot, kPairNB * 128);
        tmem_relinquish_cg<CG>();
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) cluster_sync_all();  // both CTAs' barriers initialised, TMEM allocated
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;

    if (warp == 4) {
        // ------------------------------------------------------------------ strip producer
        int it = 0;
        bool failed = false;
        const uint32_t tx = (uint32_t)(2 * p.win_srows * pitch * 128);
        for (int t = unit0; t < total_units; t += nunits, ++it) {
            const int s = it & 1;
            const uint32_t ok = mbar_wait_warp(&sempty[s], ((it >> 1) & 1) ^ 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                failed = true;
                break;
            }
            const int L0 = (t * CG + rank) * 128, g0 = L0 / pitch;
            int n = g0 / p.win_Hp, hp = g0 - n * p.win_Hp;
            // rank 1: entries between its strip and rank 0's, so that both tiles sit at rank 0's offset
            const int shift = (CG == 2 && rank == 1) ? (L0 - 128) % pitch - L0 % pitch : 0;
            uint8_t* dst = strip + 2 * s * half_bytes + (first + shift) * 128;
            uint32_t fb = smem_u32(&sfull[s]);
            if (rank == 0) mbar_arrive_expect_tx_elect(&sfull[s], CG * tx);
            if (CG == 2) fb = mapa_shared(fb, 0);
            for (int r = 0; r < p.win_srows; ++r) {
                // padded row hp of image n = row hp - 1 from pair -1 (padding rows, pair -1 and images past the
                // batch are outside the tensor and arrive as zeros)
                tma_load_5d_cg<CG>(dst + r * pitch * 128, &tmA, fb, 0, 0, -1, hp - 1, n);
                tma_load_5d_cg<CG>(dst + half_bytes + r * pitch * 128, &tmA, fb, 0, 1, -1, hp - 1, n);
                if (++hp == p.win_Hp) {
                    hp = 0;
                    ++n;
                }
            }
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            if (rank == 0) {
                for (int i = it - 1; i >= 0 && i >= it - 2; --i) (void)mbar_drain_warp(&sfull[i & 1], (i >> 1) & 1);
            } else {
                // rank 1's copies complete on rank 0's barriers: give them a fixed time instead
                const uint64_t t0 = globaltimer();
                while (globaltimer() - t0 < 1000000ull) {
                }
            }
        }
    } else if (warp == 5) {
        // ------------------------------------------------------------------ weights
        uint32_t fb = smem_u32(&wfull);
        if (rank == 0) mbar_arrive_expect_tx_elect(&wfull, (uint32_t)(CG * kWeights));
        if (CG == 2) fb = mapa_shared(fb, 0);
        if constexpr (CG == 1) {
            for (int tap = 0; tap < 9; ++tap)
                win_load_wtile<64, DG, 1>(p, &tmB, sgen + (tap / 3 * 3 + 2 - tap % 3) * BT, fb, tap, 0, 0, 0);
        } else {
            for (int r = 0; r < 3; ++r) {
                uint8_t* w = sgen + 3 * r * BT;
                tma_load_2d_cg<2>(w, &tmB, fb, (3 * r + 1 - rank) * 64, 0);
                tma_load_2d_cg<2>(w + BT, &tmB, fb, (3 * r + 2 - rank) * 64, 0);
                tma_load_2d_cg<2>(w + 2 * BT, &tmB32, fb, 3 * r * 64, 32 * rank);
                tma_load_2d_cg<2>(w + 2 * BT + BT / 2, &tmB32, fb, (3 * r + 2) * 64, 32 * rank);
            }
            tma_load_2d_cg<2>(sgen + 9 * BT, &tmB32, fb, 64, 32 * rank);
        }
        if (rank == 0) (void)mbar_drain_warp(&wfull, 0);
    } else if (warp == 6) {
        // ------------------------------------------------------------------ MMA issuer (rank 0 of a pair)
        const uint32_t id64 = idesc_act(BM * CG, 64, 0u, DG ? 1u : 0u), id128 = idesc_act(BM * CG, 128, 0u, DG ? 1u : 0u);
        const uint64_t dB = DG ? smem_desc(sbase, 8192, 1024, kSwizzle128B) : smem_desc(sbase, 16, 1024, kSwizzle128B);
        constexpr uint64_t kB = DG ? (2048 >> 4) : (32 >> 4);  // a K-step of B
        // B operands of filter row r: E[j] and O[j] (N = 128), O[j-1] and E[j+1] (N = 64); of the first
        // K-step of E[j] its two halves
        constexpr uint64_t kTap = BT >> 4;
        constexpr uint64_t kE = CG == 1 ? kTap : 0, kO = CG == 1 ? 0 : kTap, kO1 = 2 * kTap,
                           kE1 = CG == 1 ? 0 : 2 * kTap + kTap / 2, kW1 = CG == 1 ? kTap : 9 * kTap;
        int it = 0;
        bool failed = false;
        if (rank == 0) {
            const uint32_t ok = mbar_wait_warp(&wfull, 0, &abort_flag);
            failed = __any_sync(0xffffffffu, ok == 0u);
        }
        for (int t = unit0; t < total_units && rank == 0 && !failed; t += nunits, ++it) {
            const int buf = it % kPairNB, s = it & 1;
            const uint32_t ok = mbar_wait_warp(&acce_bar[buf], ((it / kPairNB) & 1) ^ 1, &abort_flag);
            const uint32_t oks = mbar_wait_warp(&sfull[s], (it >> 1) & 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u || oks == 0u)) {
                failed = true;
                break;
            }
            tc_fence_after();
            const int L0 = t * CG * 128, off = L0 - (L0 / pitch) * pitch;  // the tile's start within the strip's first row
            const uint32_t d = tmem + (uint32_t)(buf * 128);
            const uint32_t sa = smem_u32(strip + 2 * s * half_bytes) + (uint32_t)((first + off) * 128);
            const uint64_t e0 = smem_desc(sa, 16, 1024, kSwizzle128B);
            const uint64_t o0 = smem_desc(sa + (uint32_t)half_bytes, 16, 1024, kSwizzle128B);
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const uint64_t row = (uint64_t)(r * pitch * 8);  // 128-byte entries in 16-byte units
                const uint64_t w = dB + 3 * r * kTap;
                mma_act_x4_elect_cg<CG>(d, o0 + row, 2, w + kO1, kB, id64, r > 0 ? 1u : 0u);
                if (r == 0) {  // the odd pixel's first K-step does not accumulate, the even one's does
                    mma_act_elect_cg<CG>(d, e0 + 8, w + kW1, id64, 1u);
                    mma_act_elect_cg<CG>(d + 64, e0 + 8, w + kO1, id64, 0u);
#pragma unroll
                    for (int k = 1; k < 4; ++k)
                        mma_act_elect_cg<CG>(d, e0 + (uint64_t)(8 + 2 * k), w + kE + k * kB, id128, 1u);
                } else {
                    mma_act_x4_elect_cg<CG>(d, e0 + row + 8, 2, w + kE, kB, id128, 1u);
                }
                mma_act_x4_elect_cg<CG>(d, o0 + row + 8, 2, w + kO, kB, id128, 1u);
                mma_act_x4_elect_cg<CG>(d + 64, e0 + row + 16, 2, w + kE1, kB, id64, 1u);
            }
            mma_commit_elect_cg<CG>(&sempty[s], kAll);
            mma_commit_elect_cg<CG>(&accf_bar[buf], kAll);  // arrives when this unit's MMAs have completed
        }
        if (rank == 0) {
            if (failed && lane == 0) report_timeout(&abort_flag);
            mma_commit_elect_cg<CG>(&drain_bar, 1);
            (void)mbar_drain_warp(&drain_bar, 0);
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 0-3)
        float* st_tile = epi_tile + warp * 32 * 33;
        float* wsum = epi_sum + warp * 2 * 64;
        RowStats<64> rs;
        rs.zero();
        const int img = p.win_Hp * pitch;
        int it = 0;
        for (int t = unit0; t < total_units; t += nunits, ++it) {
            const int buf = it % kPairNB, tile = t * CG + rank;
            const uint32_t ok = mbar_wait_warp(&accf_bar[buf], (it / kPairNB) & 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                if (lane == 0) report_timeout(&abort_flag);
                break;
            }
            tc_fence_after();
            const int L = tile * 128 + warp * 32 + lane;
            const int n = L / img, rem = L - n * img;
            const int hp = rem / pitch, j = rem - hp * pitch;
            const bool valid = tile < p.total_tiles && n < p.gN && hp < p.win_P && j < pitch - 1;
            const int64_t out_row = ((int64_t)n * p.win_P + hp) * (pitch - 1) + j;
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(buf * 128);
            // the next chunk's TMEM load in flight while this one is converted and stored
            uint32_t va[32], vb[32];
            tmem_ld_32x32b_x32(taddr, va);
#pragma unroll
            for (int c = 0; c < 4; ++c) {  // pixel c / 2, channels 32 * (c % 2) ..
                uint32_t(&cur)[32] = (c & 1) ? vb : va;
                uint32_t(&nxt)[32] = (c & 1) ? va : vb;
                tmem_ld_wait_regs(cur);
                if (c < 3) tmem_ld_32x32b_x32(taddr + (uint32_t)((c + 1) * 32), nxt);
                float back[32];
                store_row_chunk_act(p, cur, valid, out_row, c * 32, back);
                if (want_stats) rs.add(c % 2, back);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (CG == 2)
                    mbar_arrive_cluster(mapa_shared(smem_u32(&acce_bar[buf]), 0));
                else
                    mbar_arrive(&acce_bar[buf]);
            }
        }
        if (want_stats) {
            rs.flush(st_tile, wsum, 64, 0, lane);
            asm volatile("bar.sync 1, 128;" ::: "memory");
            float* dst = p.stats + (int64_t)blockIdx.x * 128;
            const int c = threadIdx.x;
            dst[c] = (epi_sum[c] + epi_sum[128 + c]) + (epi_sum[256 + c] + epi_sum[384 + c]);
        }
    }
    tc_fence_before();
    __syncthreads();
    // neither CTA of a pair leaves while the other may still signal its barriers or read its TMEM
    if constexpr (CG == 2) cluster_sync_all();
    if (warp == 6) {
        tc_fence_after();
        tmem_dealloc_cg<CG>(tmem, kPairNB * 128);
    }
}

// ----------------------------------------------------------------------------- window weight gradient
// dW[k][r][s][c] = sum over positions L of dy[L][k] * x_pad[L + r*Wp + s][c] for stride-1 layers with
// 64 input and 64 output channels and three, four, nine or ten taps (2x2, 1x3, 1x4, 2x5, 5x2; 3x3, 3x1 and 4x1
// filters go to conv_wgrow_kernel where that can), in the padded position space
// of conv_win_kernel: dy is zero at the positions that are not outputs (its strip rows are read
// with w from 0 to Wp-1 and h from 0 to Hp-1, and the zero fill of TMA covers w >= Q and h >= P).
// A CTA owns all taps*64 x 64 outputs, as ceil(taps/2) 128 x 64 TMEM accumulators (tap pairs
// (0,1), (2,3), ...), and one contiguous range of K-blocks (256 positions, or two whole padded
// rows when those are a multiple of 16; split-K over CTAs, fixed-order reduce afterwards).  Per
// K-block it loads one x strip and one dy strip; all taps read the same x strip.  A operand (x,
// MN-major: a 128-byte strip row holds the 64 channels of one position) of tap pair (t0, t1):
// start row off(t0) + 16j for K-step j, second 64-row half LBO = (off(t1) - off(t0)) rows
// further; for an odd tap count the last pair's second half is computed and not stored.
// B operand (dy, MN-major): start row 16j.
constexpr int kWgWinKB = 256;  // positions per K-block (row-aligned K-blocks may be shorter)

template <int NACC>  // accumulators: ceil(taps / 2)
__global__ void __launch_bounds__(kWinThreads, 1)
    conv_wgwin_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmDY,
                      const ConvParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[2], empty_bar[2], accf_bar, acce_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    const int Wp = p.win_Wp;
    const int xalign = ((p.win_srows * Wp * 128 + 1023) / 1024) * 1024;  // dy strip offset in a stage
    const int stage_bytes = p.win_strip_bytes;
    const int ntaps = p.win_R * p.win_S;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&full_bar[i], 2);  // one expect_tx arrival per producer warp
            mbar_init(&empty_bar[i], 1);
        }
        mbar_init(&accf_bar, 1);
        mbar_init(&acce_bar, 4);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    if ((warp == 4 || warp == 5) && lane == 0) tma_prefetch_desc(warp == 4 ? &tmX : &tmDY);
    if (warp == 6) {
        tmem_alloc(&tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;

    if (warp == 4 || warp == 5) {
        // ------------------------------------------------------------------ producers: x rows (4), dy rows (5)
        const bool is_x = warp == 4;
        const int rows = is_x ? p.win_srows : p.win_dyrows;
        const uint32_t tx = (uint32_t)(rows * Wp * 128);
        int it = 0;
        bool failed = false;
        for (int z = blockIdx.x; z < p.zdim && !failed; z += gridDim.x) {
            const int kb0 = z * p.kb_per_split, kb1 = min(p.num_kb, kb0 + p.kb_per_split);
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                const int s = it & 1;
                const uint32_t ok = mbar_wait_warp(&empty_bar[s], ((it >> 1) & 1) ^ 1, &abort_flag);
                if (__any_sync(0xffffffffu, ok == 0u)) {
                    failed = true;
                    break;
                }
                uint8_t* dst = sgen + s * stage_bytes + (is_x ? 0 : xalign);
                const int g0 = kb * p.win_tile / Wp;
                mbar_arrive_expect_tx_elect(&full_bar[s], tx);
                for (int r = 0; r < rows; ++r) {
                    const int g = g0 + r;
                    const int n = g / p.win_Hp, hp = g - n * p.win_Hp;
                    if (is_x)
                        tma_load_4d_elect(dst + r * Wp * 128, &tmX, &full_bar[s], 0, -p.win_pw, hp - p.win_ph, n);
                    else
                        tma_load_4d_elect(dst + r * Wp * 128, &tmDY, &full_bar[s], 0, 0, hp, n);
                }
            }
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            for (int i = it - 1; i >= 0 && i >= it - 2; --i) (void)mbar_drain_warp(&full_bar[i & 1], (i >> 1) & 1);
        }
    } else if (warp == 6) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = idesc_act(BM, 64, 1u, 1u);
        // strip-row offsets of each tap pair's two halves (the unused half of an odd last pair
        // reads the row after its first half), once per CTA
        int o0[NACC], o1[NACC];
#pragma unroll
        for (int pp = 0; pp < NACC; ++pp) {
            const int t0 = 2 * pp, t1 = 2 * pp + 1;
            o0[pp] = (t0 / p.win_S) * Wp + t0 % p.win_S;
            o1[pp] = t1 < ntaps ? (t1 / p.win_S) * Wp + t1 % p.win_S : o0[pp] + 1;
        }
        int it = 0, lt = 0;
        bool failed = false;
        for (int z = blockIdx.x; z < p.zdim && !failed; z += gridDim.x, ++lt) {
            const uint32_t ok = mbar_wait_warp(&acce_bar, (lt & 1) ^ 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                failed = true;
                break;
            }
            tc_fence_after();
            const int kb0 = z * p.kb_per_split, kb1 = min(p.num_kb, kb0 + p.kb_per_split);
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                const int s = it & 1;
                const uint32_t okf = mbar_wait_warp(&full_bar[s], (it >> 1) & 1, &abort_flag);
                if (__any_sync(0xffffffffu, okf == 0u)) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                const int P0 = kb * p.win_tile;
                const int off = P0 - (P0 / Wp) * Wp;
                const uint32_t xa = sbase + (uint32_t)(s * stage_bytes), ya = xa + (uint32_t)xalign;
#pragma unroll 1
                for (int j = 0; j < p.win_tile / 16; ++j) {
                    const uint64_t bd = smem_desc(ya + (uint32_t)((off + 16 * j) * 128), 16384, 1024, kSwizzle128B);
#pragma unroll
                    for (int pp = 0; pp < NACC; ++pp) {
                        const uint64_t ad = smem_desc(xa + (uint32_t)((off + o0[pp] + 16 * j) * 128),
                                                      (uint32_t)((o1[pp] - o0[pp]) * 128), 1024, kSwizzle128B);
                        mma_act_elect(tmem + (uint32_t)(pp * 64), ad, bd, idesc, (kb > kb0 || j > 0) ? 1u : 0u);
                    }
                }
                mma_commit_elect(&empty_bar[s]);
            }
            mma_commit_elect(&accf_bar);  // arrives when this split's MMAs have completed
        }
        if (failed && lane == 0) report_timeout(&abort_flag);
        mma_commit_elect(&drain_bar);
        (void)mbar_drain_warp(&drain_bar, 0);
    } else {
        // ------------------------------------------------------------------ epilogue (warps 0-3)
        const int i = warp * 32 + lane;  // TMEM lane = accumulator row
        int lt = 0;
        for (int z = blockIdx.x; z < p.zdim; z += gridDim.x, ++lt) {
            const uint32_t ok = mbar_wait_warp(&accf_bar, lt & 1, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                if (lane == 0) report_timeout(&abort_flag);
                break;
            }
            tc_fence_after();
            const int kb0 = z * p.kb_per_split;
            const bool have_acc = min(p.num_kb, kb0 + p.kb_per_split) > kb0;
#pragma unroll 1
            for (int pp = 0; pp < NACC; ++pp) {
                const int tap = 2 * pp + (i >> 6), c = i & 63;
                const bool valid = tap < ntaps;
                const int m = tap * 64 + c;  // row of dW viewed as [k][(r, s, c)]
#pragma unroll 1
                for (int ch = 0; ch < 2; ++ch) {
                    uint32_t v[32];
                    if (have_acc) {
                        tmem_ld_32x32b_x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(pp * 64 + ch * 32), v);
                        tmem_ld_wait();
                    } else {
#pragma unroll
                        for (int k = 0; k < 32; ++k) v[k] = 0u;
                    }
                    if (valid) {
                        // [slice][k][m]: consecutive lanes hold consecutive m, one 128-byte line per store
                        float* o = static_cast<float*>(p.out) + ((int64_t)(p.zdim > 1 ? z : 0) * 64 + ch * 32) * p.M + m;
                        if (p.zdim == 1 && p.wg_accumulate) {
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] += __uint_as_float(v[k]);
                        } else {
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] = __uint_as_float(v[k]);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce_bar);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 6) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ----------------------------------------------------------------------------- row-block weight gradient
// dW[k][r][s][c] of a 3x3 stride-1 layer with 64 input and 64 output channels.  A K-block is R whole
// output rows of one image at a row pitch of `win_Wp` >= W + 2*pw positions (R * pitch a multiple of
// 16): one x strip of R + 2 padded rows from column -pw, and one dy strip of R rows from column -2, so
// that strip position h*pitch + w + n holds dy at column w + n - 2 (zeros outside the output).  Then
//     dW[r][s] = sum over L of x[L + r*pitch] * dy[L + 2 - s]
// and a column tap is a shift of dy, a row tap a shift of x.  Both are 128-byte rows of one strip
// apart, so MN-major operand atoms that overlap in shared memory (a leading-dimension step of one or
// two rows, or of one pitch) put two row taps on M and three column taps on N:
//     accumulator 0, 128 x 192: A = x rows {L, L + pitch}, B = dy rows {L, L + 1, L + 2}: taps (0..1, 2..0)
//     accumulator 1, 128 x 128: A = x rows {L + 2*pitch, + 1}, B = dy rows {L, L + 2}: taps (2, 2), (2, 0)
//                               in the first half, (2, 1) and an unused product in the second
// Two MMAs of 320 columns (160 tensor cycles) per 16 positions.  One tap pair per N = 64 MMA, five of
// them per 16 positions, is bound by their operand reads (6 KB of shared memory per 32 cycles of tensor
// time): 56x56, batch 512 and 128: 114.8 -> 94.9 us and 43.6 -> 38.0 us with the reduce; 72x72, batch
// 185 75.5 -> 59.9; 24x24, batch 512 36.3 -> 28.7; 32x32, batch 64 19.2 -> 17.4.
// Position shifts reach two rows past the dy strip and one past the x strip: those 128-byte rows
// are the next row's columns -2, -1 and -pw, which are zeros in any strip and are written here once.
// COL: an R x 1 filter (R = 3 or 4: the stems over their unrolled inputs).  A K-block is a band of
// `win_Wp` columns of several output rows: without column taps a band needs no neighbouring columns,
// and a narrow band of many rows reads few x rows twice (R - 1 per block; conv_wgwin_kernel's blocks
// of one or two whole rows read each x row two to four times from L2).  Accumulator 0 holds taps 0
// and 1 (x rows one band row apart), accumulator 1 taps 2 and 3, both 128 x 64.  Bound by memory;
// against conv_wgwin_kernel, with the reduce: 4 taps, 115x112, batch 512 277.7 -> 248.7 us (6.7 TB/s),
// 83x80 175.7 -> 136.5, 67x64 134.7 -> 92.0, batch 64 23.9 -> 17.3; 147x144, batch 185 218.4 -> 163.4;
// 3 taps, 32x32, batch 512 36.8 -> 31.6, 24x24 27.5 -> 18.0.
constexpr int kWgRowMaxStages = 4;

template <bool COL>
__global__ void __launch_bounds__(kWinThreads, 1)
    conv_wgrow_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmDY,
                      const ConvParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kWgRowMaxStages], empty_bar[kWgRowMaxStages], accf_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    const int pitch = p.win_Wp, rows = p.win_dyrows;
    const int xbytes = p.win_srows * pitch * 128, ybytes = rows * pitch * 128;
    const int xalign = p.win_margin;  // dy strip offset in a stage
    const int stage_bytes = p.win_strip_bytes, stages = p.win_stages;

    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; ++i) {
            mbar_init(&full_bar[i], 2);  // one expect_tx arrival per producer warp
            mbar_init(&empty_bar[i], 1);
        }
        mbar_init(&accf_bar, 1);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    // the zero rows behind each strip (8 16-byte words per row), before any MMA reads them
    for (int i = threadIdx.x; i < stages * 24; i += blockDim.x) {
        if (COL) break;  // no shifts
        const int s = i / 24, w = i % 24;
        uint8_t* dst = sgen + s * stage_bytes + (w < 8 ? xbytes + 16 * w : xalign + ybytes + 16 * (w - 8));
        *reinterpret_cast<uint4*>(dst) = make_uint4(0, 0, 0, 0);
    }
    fence_async_shared();
    if ((warp == 4 || warp == 5) && lane == 0) tma_prefetch_desc(warp == 4 ? &tmX : &tmDY);
    if (warp == 6) {
        tmem_alloc(&tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;
    // this CTA's K-blocks (grid = slices: at least one K-block each)
    const int z = blockIdx.x;
    const int kb0 = z * p.kb_per_split, kb1 = min(p.num_kb, kb0 + p.kb_per_split);

    if (warp == 4 || warp == 5) {
        // ------------------------------------------------------------------ producers: x strips (4), dy strips (5)
        const bool is_x = warp == 4;
        const int bpi = p.win_bpi;  // K-blocks per image
        int s = 0, it = 0;
        uint32_t phase = 1;
        bool failed = false;
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const uint32_t ok = mbar_wait_warp(&empty_bar[s], phase, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                failed = true;
                break;
            }
            uint8_t* dst = sgen + s * stage_bytes + (is_x ? 0 : xalign);
            const int n = kb / bpi, rem = kb - n * bpi;
            const int h0 = (COL ? rem / p.win_ni : rem) * rows, w0 = COL ? rem % p.win_ni * pitch : 0;
            mbar_arrive_expect_tx_elect(&full_bar[s], (uint32_t)(is_x ? xbytes : ybytes));
            if (is_x)
                tma_load_4d_elect(dst, &tmX, &full_bar[s], 0, w0 - p.win_pw, h0 - p.win_ph, n);
            else
                tma_load_4d_elect(dst, &tmDY, &full_bar[s], 0, COL ? w0 : -2, h0, n);
            if (++s == stages) {
                s = 0;
                phase ^= 1;
            }
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            for (int i = it - 1; i >= 0 && i >= it - stages; --i)
                (void)mbar_drain_warp(&full_bar[i % stages], (i / stages) & 1);
        }
    } else if (warp == 6) {
        // ------------------------------------------------------------------ MMA issuer
        constexpr uint32_t kN0 = COL ? 64 : 192, kN1 = COL ? 64 : 128;
        const uint32_t idesc0 = idesc_act(BM, kN0, 1u, 1u), idesc1 = idesc_act(BM, kN1, 1u, 1u);
        const uint64_t dA0 = smem_desc(0, (uint32_t)(pitch * 128), 1024, kSwizzle128B);
        const uint64_t dA1 = COL ? dA0 : smem_desc(0, 128, 1024, kSwizzle128B);
        const uint64_t dB0 = smem_desc(0, 128, 1024, kSwizzle128B);
        const uint64_t dB1 = smem_desc(0, 256, 1024, kSwizzle128B);
        const uint32_t row2 = (uint32_t)(2 * pitch * 8);  // two rows, in 16-byte units
        const int ksteps = p.win_tile / 16;
        bool failed = false;
        int s = 0;
        uint32_t phase = 0;
        const uint32_t ok = mbar_wait_warp(&full_bar[0], 0, &abort_flag);
        failed = __any_sync(0xffffffffu, ok == 0u);
        for (int kb = kb0; kb < kb1 && !failed; ++kb) {
            tc_fence_after();
            const uint32_t xa = ((sbase + (uint32_t)(s * stage_bytes)) >> 4) & 0x3FFFu, ya = xa + ((uint32_t)xalign >> 4);
            auto step = [&](int j, uint32_t acc) {
                const uint32_t xj = xa + (uint32_t)(j * 128), yj = ya + (uint32_t)(j * 128);  // 16 rows of 128 bytes
                mma_act_elect(tmem, dA0 + xj, dB0 + yj, idesc0, acc);
                mma_act_elect(tmem + kN0, dA1 + (xj + row2), dB1 + yj, idesc1, acc);
            };
            step(0, kb > kb0 ? 1u : 0u);
#pragma unroll 4
            for (int j = 1; j < ksteps - 1; ++j) step(j, 1u);
            const int sc = s;
            if (++s == stages) {
                s = 0;
                phase ^= 1;
            }
            // the next stage's wait while the tensor pipe still has work queued
            if (kb + 1 < kb1) {
                const uint32_t okn = mbar_wait_warp(&full_bar[s], phase, &abort_flag);
                failed = __any_sync(0xffffffffu, okn == 0u);
            }
            if (ksteps > 1) step(ksteps - 1, 1u);
            mma_commit_elect(&empty_bar[sc]);
        }
        mma_commit_elect(&accf_bar);  // arrives when this slice's MMAs have completed
        if (failed && lane == 0) report_timeout(&abort_flag);
        mma_commit_elect(&drain_bar);
        (void)mbar_drain_warp(&drain_bar, 0);
    } else {
        // ------------------------------------------------------------------ epilogue (warps 0-3)
        const int i = warp * 32 + lane;  // TMEM lane = accumulator row
        const int half = i >> 6, c = i & 63;
        const uint32_t ok = mbar_wait_warp(&accf_bar, 0, &abort_flag);
        if (__any_sync(0xffffffffu, ok == 0u)) {
            if (lane == 0) report_timeout(&abort_flag);
        } else {
            tc_fence_after();
#pragma unroll 1
            for (int b = 0; b < (COL ? 2 : 5); ++b) {  // 64-column blocks: one tap per half
                const int tap = COL     ? (2 * b + half < p.win_R ? 2 * b + half : -1)
                                : b < 3 ? half * 3 + 2 - b
                                        : half == 0 ? 6 + (b == 3 ? 2 : 0) : b == 4 ? 7 : -1;
                const int m = tap * 64 + c;  // row of dW viewed as [k][(r, s, c)]
#pragma unroll 1
                for (int ch = 0; ch < 2; ++ch) {
                    uint32_t v[32];
                    tmem_ld_32x32b_x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(b * 64 + ch * 32), v);
                    tmem_ld_wait();
                    if (tap >= 0) {
                        // [slice][k][m]: consecutive lanes hold consecutive m, one 128-byte line per store
                        float* o = static_cast<float*>(p.out) + ((int64_t)z * 64 + ch * 32) * p.M + m;
                        if (p.zdim == 1 && p.wg_accumulate) {
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] += __uint_as_float(v[k]);
                        } else {
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] = __uint_as_float(v[k]);
                        }
                    }
                }
            }
            tc_fence_before();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 6) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ----------------------------------------------------------------------------- filter-row weight gradient
// dW[k][r][s][c] of a 3x3 stride-1 layer whose channels come in 128s.  A CTA owns one filter row r,
// 128 input channels and 128 output channels (384 accumulator columns of 128 rows), and one range of
// K-blocks.  A K-block is R whole output rows of one image, or all rows of several small images, at
// a pitch of Wp = W + 2*pw positions: the x rows that filter row r reads (from column -pw) and the dy
// rows from column -2, each as two 64-channel strips.  As in conv_wgrow_kernel a column tap is a shift
// of dy by one 128-byte row, so that one MN-major B operand of three overlapping atoms holds the three
// column taps:
//     accumulator h, 128 x 192: A = x rows L (two 64-channel strips), B = dy strip h, rows {L, L + 1, L + 2}: s = 2..0
// Two N = 192 MMAs per 16 positions (192 tensor cycles) read 16 x 512 bytes that TMA loaded once, 43
// bytes per cycle, where the implicit GEMM loads x once per tap (96 bytes per cycle at 128 columns).
// The positions of a block are rounded up to 16: the rows behind the strips are zeros written once.
// Zeros of dy meet the x of their positions, as in conv_wgwin_kernel and conv_wgrow_kernel: an infinite x at a row's
// end (or in rows past a last block) makes the taps that do not read it NaN as well; the taps that do are not finite
// in any form.
// Every CTA ends with 196 KB of partial sums.  A cluster of CL CTAs (win_cl; the same outputs, CL
// consecutive K ranges) adds them before they leave the SMs: when all MMAs of the cluster are done, each
// CTA sends the 32-column chunks it does not own into the strip buffers of their owner (distributed
// shared memory, as in conv_splitk_kernel), and adds what it received in rank order.
constexpr int kWgTapMaxStages = 4;
constexpr int kWgTapThreads = 32 * 11;  // 8 epilogue warps, 2 producers, MMA

__global__ void __launch_bounds__(kWgTapThreads, 1)
    conv_wgtap_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmDY,
                      const ConvParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kWgTapMaxStages], empty_bar[kWgTapMaxStages], accf_bar, drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
    const int strip = p.win_strip_bytes;  // one 64-channel strip; a stage holds x0, x1, dy0, dy1
    const int loaded = p.win_dyrows * 128;  // bytes TMA writes of it
    const int stages = p.win_stages;

    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; ++i) {
            mbar_init(&full_bar[i], 2);  // one expect_tx arrival per producer warp
            mbar_init(&empty_bar[i], 1);
        }
        mbar_init(&accf_bar, 1);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    // the zero rows behind each strip, before any MMA reads them
    const int tail = (strip - loaded) / 16;
    for (int i = threadIdx.x; i < stages * 4 * tail; i += blockDim.x)
        *reinterpret_cast<uint4*>(sgen + (i / tail) * strip + loaded + i % tail * 16) = make_uint4(0, 0, 0, 0);
    fence_async_shared();
    if ((warp == 8 || warp == 9) && lane == 0) tma_prefetch_desc(warp == 8 ? &tmX : &tmDY);
    if (warp == 10) {
        tmem_alloc(&tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_trigger();  // a convolution launched next may start its set-up: this CTA has its TMEM
    grid_dependency_wait();  // the set-up above may overlap the previous kernel; memory only after it
    const uint32_t tmem = tmem_slot;
    // this CTA's outputs and K-blocks (possibly none): the clusters of one slice are adjacent
    const int groups = p.m_tiles * p.n_tiles;  // 3 filter rows x 128-channel blocks of x, 128-channel blocks of dy
    const int CL = p.win_cl, rank = CL > 1 ? (int)cluster_ctarank() : 0;
    const int cluster = blockIdx.x / CL, slice = cluster / groups, gi = cluster - slice * groups;
    const int z = slice * CL + rank;
    const int r = gi % 3, c0 = gi / 3 % (p.m_tiles / 3) * 128, n0 = gi / p.m_tiles * 128;
    const int kb0 = z * p.kb_per_split, kb1 = min(p.num_kb, kb0 + p.kb_per_split);

    if (warp == 8 || warp == 9) {
        // ------------------------------------------------------------------ producers: x strips (8), dy strips (9)
        const bool is_x = warp == 8;
        int s = 0, it = 0;
        uint32_t phase = 1;
        bool failed = false;
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const uint32_t ok = mbar_wait_warp(&empty_bar[s], phase, &abort_flag);
            if (__any_sync(0xffffffffu, ok == 0u)) {
                failed = true;
                break;
            }
            uint8_t* dst = sgen + (4 * s + (is_x ? 0 : 2)) * strip;
            const int i = kb / p.win_bpi, h0 = (kb - i * p.win_bpi) * p.win_srows, img = i * p.win_ni;
            if (!(p.test_stall && is_x && blockIdx.x == 0 && it == 0)) {  // stage 0 never fills (bounded-wait test)
                mbar_arrive_expect_tx_elect(&full_bar[s], (uint32_t)(2 * loaded));
                for (int h = 0; h < 2; ++h) {
                    if (is_x)
                        tma_load_4d_elect(dst + h * strip, &tmX, &full_bar[s], c0 + 64 * h, -p.win_pw, h0 + r - p.win_ph, img);
                    else
                        tma_load_4d_elect(dst + h * strip, &tmDY, &full_bar[s], n0 + 64 * h, -2, h0, img);
                }
            }
            if (++s == stages) {
                s = 0;
                phase ^= 1;
            }
        }
        if (failed) {
            if (lane == 0) report_timeout(&abort_flag);
            for (int i = it - 1; i >= 0 && i >= it - stages; --i)
                (void)mbar_drain_warp(&full_bar[i % stages], (i / stages) & 1);
        }
    } else if (warp == 10) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = idesc_act(BM, 192, 1u, 1u);
        const uint64_t dA = smem_desc(0, (uint32_t)strip, 1024, kSwizzle128B);
        const uint64_t dB = smem_desc(0, 128, 1024, kSwizzle128B);
        const uint32_t strip16 = (uint32_t)strip >> 4;
        const int ksteps = p.win_tile / 16;
        int s = 0;
        uint32_t phase = 0;
        bool failed = false;
        if (kb0 < kb1) {
            const uint32_t ok = mbar_wait_warp(&full_bar[0], 0, &abort_flag);
            failed = __any_sync(0xffffffffu, ok == 0u);
        }
        for (int kb = kb0; kb < kb1 && !failed; ++kb) {
            tc_fence_after();
            // descriptor addresses are 14 bits: in a cluster the upper bits of sbase hold the CTA's rank
            const uint32_t xa = ((sbase + (uint32_t)(4 * s * strip)) >> 4) & 0x3FFFu, ya = xa + 2 * strip16;
            auto step = [&](int j, uint32_t acc) {
                const uint32_t xj = xa + (uint32_t)(j * 128), yj = ya + (uint32_t)(j * 128);  // 16 rows of 128 bytes
                mma_act_elect(tmem, dA + xj, dB + yj, idesc, acc);
                mma_act_elect(tmem + 192, dA + xj, dB + (yj + strip16), idesc, acc);
            };
            if (ksteps > 1) step(0, kb > kb0 ? 1u : 0u);
#pragma unroll 4
            for (int j = 1; j < ksteps - 1; ++j) step(j, 1u);
            const int sc = s;
            if (++s == stages) {
                s = 0;
                phase ^= 1;
            }
            // the next stage's wait while the tensor pipe still has work queued
            if (kb + 1 < kb1) {
                const uint32_t okn = mbar_wait_warp(&full_bar[s], phase, &abort_flag);
                failed = __any_sync(0xffffffffu, okn == 0u);
            }
            step(ksteps - 1, (kb > kb0 || ksteps > 1) ? 1u : 0u);
            mma_commit_elect(&empty_bar[sc]);
        }
        mma_commit_elect(&accf_bar);  // arrives when this slice's MMAs have completed
        if (failed && lane == 0) report_timeout(&abort_flag);
        mma_commit_elect(&drain_bar);
        (void)mbar_drain_warp(&drain_bar, 0);
    } else {
        const uint32_t ok = mbar_wait_warp(&accf_bar, 0, &abort_flag);
        if (__any_sync(0xffffffffu, ok == 0u) && lane == 0) report_timeout(&abort_flag);
        tc_fence_after();
    }
    // ---------------------------------------------------------------------- epilogue (warps 0-7)
    // chunk e of 32 accumulator columns: accumulator e / 6, atom e % 6 / 2 (column tap 2 - e % 6 / 2);
    // rank q of the cluster owns chunks q * 12 / CL .., warps of one lane quarter take alternate chunks
    const int quarter = warp & 3, half = warp >> 2, own = 12 / CL;
    const int row = quarter * 32 + lane;
    const bool have_acc = kb0 < kb1;
    auto load_chunk = [&](int e, uint32_t(&v)[32]) {
        if (have_acc) {
            tmem_ld_32x32b_x32(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(e * 32), v);
            tmem_ld_wait_regs(v);
        } else {
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] = 0u;
        }
    };
    const int part = own * 128 * 32 * 4;  // bytes one CTA sends to another: [chunk][8 x float4][128 rows]
    if (CL > 1) {
        __syncwarp();
        cluster_sync_all();  // every CTA's MMAs are done: the strips may be overwritten
        if (warp < 8) {
#pragma unroll 1
            for (int i = half; i < 12 - own; i += 2) {
                const int e = (rank * own + own + i) % 12, to = e / own;
                const int slot = rank < to ? rank : rank - 1;
                const uint32_t dst = mapa_shared(sbase, (uint32_t)to) + (uint32_t)(slot * part + (e - to * own) * 16384 + row * 16);
                uint32_t v[32];
                load_chunk(e, v);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    st_cluster_v4(dst + (uint32_t)(k * 2048), v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
            }
        }
        __syncwarp();
        cluster_sync_all();  // the parts have arrived
    }
    if (warp < 8) {
        float* out = static_cast<float*>(p.out) + (int64_t)slice * p.Ncols * p.M;
#pragma unroll 1
        for (int i = half; i < own; i += 2) {
            const int e = rank * own + i;
            uint32_t v[32];
            load_chunk(e, v);
            const float4* src = reinterpret_cast<const float4*>(sgen + i * 16384 + row * 16);
            for (int q = 0; q < CL - 1; ++q)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 f = src[q * (part / 16) + k * 128];
                    v[4 * k] = __float_as_uint(__uint_as_float(v[4 * k]) + f.x);
                    v[4 * k + 1] = __float_as_uint(__uint_as_float(v[4 * k + 1]) + f.y);
                    v[4 * k + 2] = __float_as_uint(__uint_as_float(v[4 * k + 2]) + f.z);
                    v[4 * k + 3] = __float_as_uint(__uint_as_float(v[4 * k + 3]) + f.w);
                }
            // [slice][k][m]: consecutive lanes hold consecutive m, one 128-byte line per store
            const int m = (r * 3 + 2 - e % 6 / 2) * p.Cin + c0 + row;
            float* o = out + (int64_t)(n0 + e / 6 * 64 + e % 2 * 32) * p.M + m;
            if (p.zdim == 1 && p.wg_accumulate) {
#pragma unroll
                for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] += __uint_as_float(v[k]);
            } else {
#pragma unroll
                for (int k = 0; k < 32; ++k) o[(int64_t)k * p.M] = __uint_as_float(v[k]);
            }
        }
        tc_fence_before();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 10) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ----------------------------------------------------------------------------- reductions
// Per-output-channel sums of the conv epilogue's per-CTA partials part[nparts][2][K]
// (partials_colsum, fixed order).
__global__ void __launch_bounds__(kPartialsThreads) stats_reduce_kernel(const float* __restrict__ part, int nparts, int K,
                                                           float* __restrict__ sum, float* __restrict__ sumsq)
{
    float s, q;
    const int c = partials_colsum(part, nparts, K, s, q);
    if (c >= 0) {
        sum[c] = s;
        sumsq[c] = q;
    }
}

// dw[i] (+)= sum over slices of part[slice][i] in a fixed order; i runs over
// the KRSC weight gradient (the slices are already in that layout).  LANES
// threads share one float4 of dw: thread j sums slices j, j+LANES, ... (U
// loads in flight, the last round's too), then a fixed shuffle tree adds the LANES partial sums.
// LANES = 1 for a few slices, 8 for many (the 64-channel layers split K over all SMs).  A thread's chain of load
// rounds bounds it: four loads a round and a remainder one by one were seven rounds of 152 slices' 19 per
// thread, eight with the remainder together three; weight gradient and reduce 28x28x128, batch 512 79.1 -> 78.1 us,
// 16x16x128, batch 64 16.4 -> 15.9, a 14x14 projection 256 -> 512, batch 128 12.8 -> 12.2; the same bits.
// Few slices (LANES = 1) keep four loads a round, as half of eight would be empty: 16x16, 256 -> 512 stride 2, batch 64
// 16.9 -> 16.6 us.
template <int LANES>
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float* __restrict__ part, int slices, int64_t n,
                                                           float* __restrict__ dw, int accumulate)
{
    dbl::dev::grid_dependency_trigger();  // a convolution launched next may start its set-up
    constexpr int U = LANES == 1 ? 4 : 8;
    const int j = threadIdx.x % LANES;
    const int64_t n4 = n >> 2;
    const int64_t groups = blockDim.x / LANES;
    // the loop bound is the same for the whole block, so every shuffle sees all 32 lanes
    for (int64_t base = (int64_t)blockIdx.x * groups; base < n4; base += (int64_t)gridDim.x * groups) {
        const int64_t i = base + threadIdx.x / LANES;
        const int sl = i < n4 ? slices : 0;  // groups past the end add nothing and store nothing
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = j; s < sl; s += U * LANES) {
            float4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (s + u * LANES < sl)
                    v[u] = __ldcs(reinterpret_cast<const float4*>(part + (int64_t)(s + u * LANES) * n) + i);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (s + u * LANES < sl) {
                    acc.x += v[u].x;
                    acc.y += v[u].y;
                    acc.z += v[u].z;
                    acc.w += v[u].w;
                }
        }
#pragma unroll
        for (int o = LANES / 2; o; o >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o, LANES);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o, LANES);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o, LANES);
            acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o, LANES);
        }
        if (j == 0 && i < n4) {
            float4* d = reinterpret_cast<float4*>(dw) + i;
            if (accumulate) {
                const float4 o = *d;
                acc.x += o.x;
                acc.y += o.y;
                acc.z += o.z;
                acc.w += o.w;
            }
            *d = acc;
        }
    }
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = (n4 << 2) + t; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float acc = 0.f;
        for (int s = 0; s < slices; ++s) acc += part[(int64_t)s * n + i];
        dw[i] = accumulate ? dw[i] + acc : acc;
    }
}

// ----------------------------------------------------------------------------- host side
struct Plan {
    int mode;
    int BN;
    int cg = 1;          // conv_igemm_kernel CTAs per tile (2: CTA pairs with M = 256 MMAs)
    int sk = 1;          // conv_splitk_kernel CTA pairs per tile (forward and data gradient)
    ConvParams p;
    size_t ws_main = 0;  // bytes: fwd channel-sum partials, or wgrad split-K slices
    bool win = false;    // conv_win_kernel (3x3 stride-1 correlation over padded strips)
    bool res = false;    // window kernel with all weights resident in shared memory
    bool winpair = false;  // conv_winpair_kernel (64 to 64 channels, even rows)
    bool wgrow = false;  // conv_wgrow_kernel (3x3 stride-1 weight gradient, 64 channels)
    bool wgband = false; // conv_wgrow_kernel<true> (R x 1 weight gradient, 64 channels)
    bool wgtap = false;  // conv_wgtap_kernel (3x3 stride-1 weight gradient, multiples of 128 channels)
    size_t smem = 0;     // window kernel dynamic shared memory
};



int out_dim(int in, int k, int st, int pad) { return (in + 2 * pad - k) / st + 1; }

int fwd_tile_rows(int BN);

int choose_bn(int cols)
{
    if (cols % 256 == 0) return 256;
    if (cols % 128 == 0) return 128;
    return 64;
}

// Strides and pads per axis (stride_w == 0 means: the same as along H).
struct Geom {
    int sh, sw, ph, pw;
};

Geom geom(const dbl_conv_shape* s)
{
    Geom g{s->stride, s->stride_w ? s->stride_w : s->stride, s->pad, s->stride_w ? s->pad_w : s->pad};
    return g;
}

int validate(const dbl_conv_shape* s, const char* who)
{
    using dbl::set_error;
    if (!s) return set_error(DBL_ERR_INVALID, "%s: null shape", who);
    const Geom g = geom(s);
    if (s->n <= 0 || s->h <= 0 || s->w <= 0 || s->c <= 0 || s->k <= 0 || s->r <= 0 || s->s <= 0 || g.sh <= 0 ||
        g.sw <= 0 || g.ph < 0 || g.pw < 0)
        return set_error(DBL_ERR_INVALID, "%s: non-positive dimension", who);
    if (s->c % 8) return set_error(DBL_ERR_INVALID, "%s: channels must be a multiple of 8", who);
    if (s->k % 64) return set_error(DBL_ERR_UNSUPPORTED, "%s: output channels must be a multiple of 64", who);
    if (s->k > kMaxNcols || s->c > kMaxNcols * 8)
        return set_error(DBL_ERR_UNSUPPORTED, "%s: at most %d output channels", who, kMaxNcols);
    if (g.sh > 2 || g.sw > 2 || s->r > 8 || s->s > 8 || g.ph > 3 || g.pw > 3)
        return set_error(DBL_ERR_UNSUPPORTED, "%s: stride <= 2, filter <= 8, pad <= 3 per axis supported", who);
    if (out_dim(s->h, s->r, g.sh, g.ph) <= 0 || out_dim(s->w, s->s, g.sw, g.pw) <= 0)
        return set_error(DBL_ERR_INVALID, "%s: empty output", who);
    return DBL_OK;
}

// Split-K slices of the implicit-GEMM weight gradient: the count that minimises the
// modelled time of the persistent grid on a 152-SM GPU, where the busiest CTA runs
// ceil(units / 152) units of (K-blocks per slice + ~2 K-blocks of epilogue) and the
// fixed-order reduce afterwards reads every slice (one K-block of a 128 x BN tile is
// ~4 BN tensor cycles, in which the GPU streams ~10.5 KB x BN).  At least 4 K-blocks
// (512 pixels) per slice.  A fixed function of the shape, so the summation order, and
// with it the result, does not depend on the device the plan runs on.
int wgrad_splits(int tiles, int num_kb, int rows, int cols, int BN, int cg)
{
    const int kPlanSMs = 152 / cg;  // tile processors: SMs, or SM pairs
    const double slice_cost = (double)rows * cols * 4 / (10.5e3 * BN);  // K-block times to reduce one slice
    int best = 1;
    double best_cost = 1e300;
    const int max_splits = std::max(1, num_kb / 4);
    for (int sp = 1; sp <= max_splits; ++sp) {
        const int kbs = (num_kb + sp - 1) / sp;
        const int eff = (num_kb + kbs - 1) / kbs;  // slices actually used
        if (eff != sp) continue;
        const int rounds = (tiles * sp + kPlanSMs - 1) / kPlanSMs;
        const double cost = rounds * (kbs + 2.0) + (sp > 1 ? sp * slice_cost : 0.0);
        if (cost < best_cost) {
            best_cost = cost;
            best = sp;
        }
    }
    return best;
}

// Persistent grid: one CTA per SM (the kernel uses ~225 KB of shared memory), never more
// CTAs than tiles, never more than kMaxGrid (the workspace is sized for that bound).
int grid_size(int total_tiles)
{
    int g = dbl::sm_count();
    if (g > kMaxGrid) g = kMaxGrid;
    if (g > total_tiles) g = total_tiles;
    return g < 1 ? 1 : g;
}

// Dynamic shared memory the window kernel may use (227 KB per CTA, less the
// static barriers and 1 KB of alignment slack).
constexpr size_t kWinSmemMax = 232448 - 2048;

// Least dynamic shared memory of a cluster kernel: more than half of an SM's 228 KB with the block's own 1 KB, so
// that no SM holds two of their CTAs. Each takes TMEM for itself, and with two of different clusters on an SM each
// cluster could hold the columns that the other's CTA waits for, before a cluster barrier that none would pass.
constexpr size_t kClusterSmem = 117 * 1024;
static_assert(2 * (kClusterSmem + 1024) > 228 * 1024, "one CTA per SM");

// Positions per tile of the window kernels: 256 (any start), or, for rows of at
// least 64 positions, the whole rows that fit in 256 (row-aligned starts need no
// strip row for a misaligned start).
int win_tile_positions(int Wp) { return Wp >= 64 ? (kWinBMT / Wp) * Wp : kWinBMT; }

bool win_pairs();
int cta_pair_level();

// Pixel-pair window kernel (conv_winpair_kernel): 3x3, stride 1, pad 1, 64 to 64 channels, even rows whose
// two stages fit in shared memory beside the weights (W <= 98).  CTA pairs for the forward pass only
// with DBL_CONV_CTA_PAIRS=2 (56x56, batch 512 114 us against 91: the two CTAs' loads and epilogues wait for each
// other).
bool winpair_setup(const dbl_conv_shape* s, bool dgrad, Plan& pl)
{
    const Geom g = geom(s);
    if (g.sh != 1 || g.sw != 1 || s->r != 3 || s->s != 3 || g.ph != 1 || g.pw != 1) return false;
    if (s->c != 64 || s->k != 64 || (s->w & 1) || s->w < 8) return false;
    const int pitch = s->w / 2 + 1, Hp = s->h + 2;
    const int64_t L = (int64_t)s->n * Hp * pitch;
    if (pitch > 256 || L > INT32_MAX / 8) return false;
    // entries one tile's 128 accumulator rows read: start offset within a row, plus 127, plus the last tap's
    const int rows = (pitch - 1 + 127 + 2 * pitch + 2) / pitch + 1;
    int cg = !dgrad && cta_pair_level() == 2 ? 2 : 1, half = 0;
    size_t smem = 0;
    for (;; cg = 1) {
        half = ((rows + (cg == 2)) * pitch * 128 + 1023) / 1024 * 1024;  // pairs: rank 1's shift, one row in all
        smem = (cg == 2 ? 77 * 1024 : 72 * 1024) + 4 * (size_t)half + 4 * 2 * 64 * 4 + 1024;
        if (smem <= kWinSmemMax && 4 * (size_t)half >= 4 * 32 * 33 * 4) break;
        if (cg == 1) return false;
    }
    ConvParams& p = pl.p;
    pl.win = pl.winpair = pl.res = true;
    pl.BN = 64;
    pl.cg = cg;
    pl.smem = cg == 2 ? std::max(smem, kClusterSmem) : smem;
    p.win_margin = 128 % pitch;
    p.win_R = p.win_S = 3;
    p.win_ph = p.win_pw = 1;
    p.win_P = s->h;
    p.win_Q = s->w;
    p.win_Hp = Hp;
    p.win_Wp = pitch;
    p.win_tile = 128;
    p.win_srows = rows;
    p.win_strip_bytes = half;
    p.M = s->n * s->h * s->w;
    p.m_tiles = (int)((L + 127) / 128);
    p.n_tiles = 1;
    p.cblocks = 1;
    p.gN = s->n;
    p.Ncols = 64;
    p.ldo = 128;  // a row of the output is a pair of pixels
    p.Cin = 64;
    return true;
}

// Window-kernel eligibility and geometry (see conv_win_kernel): stride 1 on both
// axes, 64-channel blocks of the reduced operand (red_c), 64 or 128 output
// channels, padded rows of 10..256 positions; the data gradient (dgrad) for
// 3x3 filters with pad 1 only (its taps are the forward taps flipped).
bool win_setup(const dbl_conv_shape* s, int red_c, int out_c, bool dgrad, Plan& pl)
{
    const Geom g = geom(s);
    if (g.sh != 1 || g.sw != 1) return false;
    if (dgrad && (s->r != 3 || s->s != 3 || g.ph != 1 || g.pw != 1)) return false;
    if (s->r * s->s > 16 || red_c % 64 != 0 || (out_c != 64 && out_c != 128)) return false;
    const int Wp = s->w + 2 * g.pw, Hp = s->h + 2 * g.ph;
    if (Wp < 10 || Wp > 256) return false;
    const int P = Hp - s->r + 1, Q = Wp - s->s + 1;
    if (P <= 0 || Q <= 0) return false;
    const int64_t L = (int64_t)s->n * Hp * Wp;
    if (L > INT32_MAX / 4) return false;
    const int tile = win_tile_positions(Wp);
    // rows one tile's 256 accumulator rows read: start offset within a row, plus 255, plus the last tap's offset
    const int max_index = (tile % Wp == 0 ? 0 : Wp - 1) + kWinBMT - 1 + (s->r - 1) * Wp + (s->s - 1);
    const int srows = max_index / Wp + 1;
    const int strip = ((srows * Wp * 128 + 1023) / 1024) * 1024;
    const int BN = out_c, CB = red_c / 64, ntaps = s->r * s->s;
    const bool res = BN == 64 && CB == 1 && ntaps <= 9;
    // CTA pairs for 128-column tiles: each SM stages half of the weights; rank 1's strip is
    // shifted by up to a padded row either way, so each strip buffer gets a margin of one padded
    // row on both sides (single CTAs when the pair layout does not fit in shared memory).  The
    // 64-column forward pass with resident weights runs on pairs only with DBL_CONV_CTA_PAIRS=2:
    // it halves each SM's weight reads (a sixth of its tensor-core shared-memory reads) but
    // couples the two CTAs' loads and epilogues; with two accumulator buffers it measured slower
    // (layer1 forward at batch 384: 113 against 97 us), with four the same (122 against 123 us
    // at batch 512).
    if ((size_t)srows * Wp * 128 >= (1u << 20)) return false;
    const int epi = out_c == 64 ? WinCfg<64>::EPI : WinCfg<128>::EPI;
    int cg = win_pairs() && (BN == 128 || (BN == 64 && res && !dgrad && cta_pair_level() == 2)) ? 2 : 1;
    int margin = 0;
    size_t smem = 0;
    for (;; cg = 1) {
        margin = cg == 2 ? (Wp * 128 + 1023) / 1024 * 1024 : 0;
        const int b_bytes = (res ? ntaps * CB * WinCfg<64>::B_TILE : kWinBStages * BN * 128) / cg;
        // epilogue statistics: per-warp channel sums after the strips (the warps' transposes reuse the strips)
        const size_t strips = 2 * ((size_t)strip + 2 * (size_t)margin);
        smem = (size_t)b_bytes + strips + (size_t)epi * 2 * out_c * 4 + 1024;
        if (strips >= (size_t)epi * 32 * 33 * 4 && smem <= kWinSmemMax) break;
        if (cg == 1) return false;
    }
    ConvParams& p = pl.p;
    pl.win = true;
    pl.res = res;
    pl.BN = BN;
    pl.cg = cg;
    pl.smem = cg == 2 ? std::max(smem, kClusterSmem) : smem;
    p.win_margin = margin;
    p.win_R = s->r;
    p.win_S = s->s;
    p.win_ph = g.ph;
    p.win_pw = g.pw;
    p.win_P = P;
    p.win_Q = Q;
    p.win_Hp = Hp;
    p.win_Wp = Wp;
    p.win_tile = tile;
    p.win_srows = srows;
    p.win_strip_bytes = strip;
    p.M = s->n * P * Q;
    p.m_tiles = (int)((L + tile - 1) / tile);
    p.n_tiles = 1;
    p.cblocks = CB;
    p.gN = s->n;
    p.Ncols = out_c;
    p.ldo = out_c;
    p.Cin = red_c;
    return true;
}

// Row-block weight-gradient eligibility and geometry (see conv_wgrow_kernel): 3x3 filters at stride 1,
// 64 input and 64 output channels.  The row pitch and the rows per K-block minimise the modelled time
// of the busiest CTA: per K-block the longer of its MMAs (160 cycles per 16 positions) and its loads
// (the real columns of R + 2 x rows and R dy rows at 40 bytes per cycle), and ~100 cycles of hand-over.
bool wgrow_setup(const dbl_conv_shape* s, Plan& pl)
{
    const Geom g = geom(s);
    if (g.sh != 1 || g.sw != 1 || s->r != 3 || s->s != 3 || s->c != 64 || s->k != 64) return false;
    const int Wp = s->w + 2 * g.pw, P = s->h + 2 * g.ph - 2, Q = Wp - 2;
    if (Wp < 10 || P <= 0 || Q <= 0) return false;
    const int sms = 152;  // a fixed count: the split must not depend on the device
    int64_t best = INT64_MAX;
    ConvParams& p = pl.p;
    for (int pitch = Wp; pitch < Wp + 16 && pitch <= 256; ++pitch)
        for (int R = 1; R <= 16; ++R) {
            if ((R * pitch) % 16) continue;
            const int xalign = ((R + 2) * pitch * 128 + 128 + 1023) / 1024 * 1024;
            const int stage = xalign + (R * pitch * 128 + 256 + 1023) / 1024 * 1024;
            const int stages = std::min<int>(kWgRowMaxStages, (int)((kWinSmemMax - 1024) / stage));
            if (stages < 2) continue;
            const int64_t blocks = (int64_t)s->n * ((P + R - 1) / R);
            if (blocks > INT32_MAX / 4) continue;
            const int64_t mma = (int64_t)R * pitch * 10, load = (int64_t)(2 * R + 2) * s->w * 128 / 40;
            const int64_t cost = (blocks + sms - 1) / sms * (std::max(mma, load) + 100);
            if (cost >= best) continue;
            best = cost;
            p.win_Wp = pitch;
            p.win_dyrows = R;
            p.win_srows = R + 2;
            p.win_tile = R * pitch;
            p.win_margin = xalign;
            p.win_strip_bytes = stage;
            p.win_stages = stages;
            p.win_bpi = (P + R - 1) / R;
            p.num_kb = (int)blocks;
            pl.smem = (size_t)stages * stage + 1024;
        }
    if (best == INT64_MAX) return false;
    pl.win = pl.wgrow = true;
    pl.BN = 64;
    pl.mode = p.mode = kWgrad;
    p.win_R = p.win_S = 3;
    p.win_ph = g.ph;
    p.win_pw = g.pw;
    p.win_P = P;
    p.win_Q = Q;
    p.M = 9 * 64;
    p.Ncols = 64;
    p.m_tiles = p.n_tiles = 1;
    p.gN = s->n;
    // one contiguous range of K-blocks per CTA
    const int splits = std::min(p.num_kb, sms);
    p.kb_per_split = (p.num_kb + splits - 1) / splits;
    p.zdim = (p.num_kb + p.kb_per_split - 1) / p.kb_per_split;
    pl.ws_main = p.zdim > 1 ? (size_t)p.zdim * p.M * 64 * sizeof(float) : 0;
    return true;
}

// Filter-row weight-gradient eligibility and geometry (see conv_wgtap_kernel): 3x3 filters at stride 1,
// input and output channels in 128s.  The K-block (rows of an image, or whole images) and the number of
// K ranges, and the CTAs per cluster, minimise the modelled time of the busiest CTA on a 152-SM GPU, in
// tensor cycles: 192 per 16 positions and ~150 of hand-over per K-block, ~4000 of set-up and ~3000 of
// stores per CTA, ~9000 for sending all partial sums to other SMs (22 bytes per cycle), and the launch
// and the traffic of the fixed-order reduce of the slices.
bool wgtap_setup(const dbl_conv_shape* s, Plan& pl)
{
    const Geom g = geom(s);
    if (g.sh != 1 || g.sw != 1 || s->r != 3 || s->s != 3 || s->c % 128 || s->k % 128) return false;
    const int Wp = s->w + 2 * g.pw, P = s->h + 2 * g.ph - 2;
    if (P <= 0 || Wp <= 2 || Wp > 256) return false;
    // CTAs that 152 SMs hold in clusters of 1..4: fixed counts, the split must not depend on the device
    static const int resident[5] = {0, 152, 152, 108, 144};
    constexpr double kExchange = 9000.0, kReduce = 4000.0, kReduceSlice = 0.0030;
    constexpr int kMaxPos = 208;
    const int groups = 3 * (s->c / 128) * (s->k / 128);
    if (groups > 12) return false;  // see below
    int max_cl = 1;
    while (max_cl < 4 && dbl::cluster_held<conv_wgtap_kernel>(max_cl + 1, kWgTapThreads, kWinSmemMax)) ++max_cl;
    const int64_t elems = (int64_t)9 * s->c * s->k;
    // positions a CTA adds up: no more than the implicit GEMM (the tensor core's sums lose with their steps)
    const int BN = choose_bn(s->k), cg = 2;
    const int64_t pix = (int64_t)s->n * P * (Wp - 2), igemm_kb = (pix + 127) / 128;
    if (igemm_kb > INT32_MAX / 2) return false;
    const int igemm_splits = wgrad_splits((9 * s->c + cg * BM - 1) / (cg * BM) * (s->k / BN), (int)igemm_kb, 9 * s->c, s->k, BN, cg);
    const int64_t longest = (igemm_kb + igemm_splits - 1) / igemm_splits * 128;
    double best = 1e300;
    ConvParams& p = pl.p;
    for (int u = 1; u <= kMaxPos; ++u) {  // u rows of an image, then u - P + 1 images
        const int R = std::min(u, P), ni = std::max(1, u - P + 1);
        const int pos = ni * R * Wp;
        if (pos > kMaxPos || ni > 256) break;
        const int ksteps = (pos + 15) / 16;
        const int strip = ((ksteps * 16 + 2) * 128 + 1023) / 1024 * 1024;
        const int stages = std::min<int>(kWgTapMaxStages, (int)((kWinSmemMax - 1024) / (4 * strip)));
        if (stages < 2) break;
        const int64_t blocks = ni > 1 ? (s->n + ni - 1) / ni : (int64_t)s->n * ((P + R - 1) / R);
        if (blocks > INT32_MAX / 4) continue;
        for (int cl = 1; cl <= max_cl; ++cl)
            for (int sixth = 18, last = 0; sixth >= 1; --sixth) {  // three rounds of the slices that fit, or fewer
                int slices = std::max(1, resident[cl] / (groups * cl) * sixth / 6);
                const int64_t kbs = (blocks + slices * cl - 1) / (slices * cl);
                slices = (int)((blocks + cl * kbs - 1) / (cl * kbs));  // no cluster without a K-block
                if (slices == last) continue;
                last = slices;
                const int sp = slices * cl;
                if (kbs * ksteps * 16 > longest) continue;
                if (cl > 1 && (size_t)stages * 4 * strip < (size_t)(cl - 1) * (12 / cl) * 16384) break;
                const int rounds = (groups * sp + resident[cl] - 1) / resident[cl];
                if (rounds > 1 && ksteps < 11) continue;  // see below
                const double cost = rounds * (kbs * (ksteps * 192.0 + 150.0) + 4000.0 + 3000.0 / cl +
                                              (cl > 1 ? 2000.0 + kExchange * (cl - 1) / cl : 0.0)) +
                                    (slices > 1 ? kReduce + kReduceSlice * elems * slices : 0.0);
                if (cost >= best) continue;
                best = cost;
                p.win_Wp = Wp;
                p.win_srows = R;
                p.win_ni = ni;
                p.win_bpi = ni > 1 ? 1 : (P + R - 1) / R;
                p.win_dyrows = pos;
                p.win_tile = ksteps * 16;
                p.win_strip_bytes = strip;
                p.win_stages = stages;
                p.win_cl = cl;
                p.num_kb = (int)blocks;
                p.kb_per_split = (int)kbs;
                p.zdim = slices;
                pl.smem = (size_t)stages * 4 * strip + 1024;
            }
    }
    if (best == 1e300) return false;
    // Against the implicit GEMM (kernel and reduce, us): 28x28x128, batch 512 120 -> 81 and 128 39.0 -> 33.4;
    // 14x14x256, batch 512 91.3 -> 77.0 and 128 30.9 -> 30.4; 12x12x128, batch 512 32.0 -> 30.9.  It stays
    // the better one where the padding of a block's positions costs more than a fifth of them (10x10x256,
    // batch 128 21.4 -> 23.6), where a CTA's K range is shorter than ~22,000 tensor cycles (12x12x128, batch
    // 128 16.7 -> 18.0) and for 512 x 512 channels, whose 48 tiles leave three ranges (7x7, batch 512, three
    // slices without clusters 91.6 -> 94.6).  Large maps of 256 channels run in up to three rounds, whose ranges are
    // as short as the implicit GEMM's: 48x48, batch 219 418 -> 364 and error of dw against 64 bits 2.3e-5 -> 1.7e-5
    // (one round 334 and 5.2e-5); short K-blocks lose there (16x16, batch 2330, 144 positions 485 -> 532).
    const double used = (double)s->n * P * (Wp - 2) / ((double)p.num_kb * p.win_tile);
    if (used < 0.8 || (double)p.kb_per_split * p.win_tile * 12 < 22000.0) return false;
    if (p.win_cl > 1) pl.smem = std::max(pl.smem, kClusterSmem);
    pl.win = pl.wgtap = true;
    pl.BN = 128;
    pl.mode = p.mode = kWgrad;
    p.win_R = p.win_S = 3;
    p.win_ph = g.ph;
    p.win_pw = g.pw;
    p.M = 9 * s->c;
    p.Ncols = s->k;
    p.Cin = s->c;
    p.m_tiles = 3 * (s->c / 128);
    p.n_tiles = s->k / 128;
    p.gN = s->n;
    pl.ws_main = p.zdim > 1 ? (size_t)p.zdim * p.M * s->k * sizeof(float) : 0;
    return true;
}

// Band weight-gradient eligibility and geometry (conv_wgrow_kernel<true>): R x 1 filters, R = 3 or 4, at stride 1
// without padding along W, 64 input and 64 output channels.  The band width and rows minimise the modelled time
// of the busiest CTA: per K-block the longer of its MMAs (108 cycles per 16 positions) and its loads (40 bytes
// per cycle), and ~100 cycles of hand-over.
bool wgband_setup(const dbl_conv_shape* s, Plan& pl)
{
    const Geom g = geom(s);
    if (g.sh != 1 || g.sw != 1 || g.pw != 0 || s->s != 1 || (s->r != 3 && s->r != 4) || s->c != 64 || s->k != 64)
        return false;
    const int P = s->h + 2 * g.ph - s->r + 1;
    if (P <= 0) return false;
    const int sms = 152;  // a fixed count: the split must not depend on the device
    double best = 1e300;
    ConvParams& p = pl.p;
    for (int bands = 1; bands <= (s->w + 7) / 8; ++bands) {
        const int bw = (s->w + bands - 1) / bands;
        if (bw > 256 || (bands > 1 && bw == (s->w + bands - 2) / (bands - 1))) continue;
        for (int R = 1; R <= 32 && R < P + 16; ++R) {
            const int xrows = R + s->r - 1;
            if ((R * bw) % 16 || R * bw > 512) continue;
            const int xalign = (xrows * bw * 128 + 1023) / 1024 * 1024;
            const int stage = xalign + (R * bw * 128 + 1023) / 1024 * 1024;
            const int stages = std::min<int>(kWgRowMaxStages, (int)((kWinSmemMax - 1024) / stage));
            // with three taps the unused half of accumulator 1 reads one band row past the x strip: into the dy strip
            if (stages < 2 || (s->r == 3 && xalign + R * bw * 128 < (R + 3) * bw * 128)) continue;
            const int64_t bpi = (int64_t)bands * ((P + R - 1) / R), blocks = s->n * bpi;
            if (blocks > INT32_MAX / 4) continue;
            const double mma = R * bw * 6.75, load = (double)(xrows + R) * bw * 128 / 40.0;
            const double cost = (double)((blocks + sms - 1) / sms) * (std::max(mma, load) + 100.0);
            if (cost >= best) continue;
            best = cost;
            p.win_Wp = bw;
            p.win_dyrows = R;
            p.win_srows = xrows;
            p.win_tile = R * bw;
            p.win_margin = xalign;
            p.win_strip_bytes = stage;
            p.win_stages = stages;
            p.win_bpi = (int)bpi;
            p.win_ni = bands;
            p.num_kb = (int)blocks;
            pl.smem = (size_t)stages * stage + 1024;
        }
    }
    if (best == 1e300) return false;
    pl.win = pl.wgband = true;
    pl.BN = 64;
    pl.mode = p.mode = kWgrad;
    p.win_R = s->r;
    p.win_S = 1;
    p.win_ph = g.ph;
    p.win_pw = 0;
    p.win_P = P;
    p.win_Q = s->w;
    p.M = s->r * 64;
    p.Ncols = 64;
    p.m_tiles = p.n_tiles = 1;
    p.gN = s->n;
    // one contiguous range of K-blocks per CTA
    const int splits = std::min(p.num_kb, sms);
    p.kb_per_split = (p.num_kb + splits - 1) / splits;
    p.zdim = (p.num_kb + p.kb_per_split - 1) / p.kb_per_split;
    pl.ws_main = p.zdim > 1 ? (size_t)p.zdim * p.M * 64 * sizeof(float) : 0;
    return true;
}

// Window weight-gradient eligibility and geometry (see conv_wgwin_kernel):
// stride 1, 64 input and 64 output channels, three, four, nine or ten taps that wgrow_setup and wgband_setup do not
// take, padded rows of 10..256 positions.  As implicit GEMMs 2x5 and 5x2 filters at 56x56, batch 128 took 56 to 59 us
// instead of 43 to 44, with five times the rounding error (a K range per CTA pair instead of per CTA).
bool wgwin_setup(const dbl_conv_shape* s, Plan& pl)
{
    const Geom g = geom(s);
    if (g.sh != 1 || g.sw != 1) return false;
    if (s->c != 64 || s->k != 64) return false;
    const int ntaps = s->r * s->s;
    if ((ntaps + 1) / 2 != 2 && (ntaps + 1) / 2 != 5) return false;  // the instantiated accumulator counts
    const int Wp = s->w + 2 * g.pw, Hp = s->h + 2 * g.ph;
    if (Wp < 10 || Wp > 256) return false;
    const int P = Hp - s->r + 1, Q = Wp - s->s + 1;
    if (P <= 0 || Q <= 0) return false;
    const int64_t L = (int64_t)s->n * Hp * Wp;
    if (L > INT32_MAX / 4) return false;
    // K-block: two whole padded rows when that is a multiple of 16 positions (no misaligned start), else 256
    // (one row of 129 to 256 positions instead: 1x3 and 1x4 at 145x144, batch 32 40.1 -> 42.9 and 40.5 -> 43.5 us)
    const int kb = (Wp >= 64 && 2 * Wp <= kWgWinKB && (2 * Wp) % 16 == 0) ? 2 * Wp : kWgWinKB;
    const int start = kb % Wp == 0 ? 0 : Wp - 1;
    auto off = [&](int t) { return (t / s->s) * Wp + t % s->s; };
    const int last = (ntaps % 2) ? off(ntaps - 1) + 1 : off(ntaps - 1);  // the unused half of an odd last pair
    const int xrows = (start + kb - 1 + last) / Wp + 1;
    const int dyrows = (start + kb - 1) / Wp + 1;
    const int xalign = ((xrows * Wp * 128 + 1023) / 1024) * 1024;
    const int stage = xalign + ((dyrows * Wp * 128 + 1023) / 1024) * 1024;
    const size_t smem = 2 * (size_t)stage + 1024;
    if (smem > kWinSmemMax) return false;
    ConvParams& p = pl.p;
    pl.win = true;
    pl.BN = 64;
    pl.smem = smem;
    pl.mode = p.mode = kWgrad;
    p.win_R = s->r;
    p.win_S = s->s;
    p.win_ph = g.ph;
    p.win_pw = g.pw;
    p.win_P = P;
    p.win_Q = Q;
    p.win_Hp = Hp;
    p.win_Wp = Wp;
    p.win_tile = kb;
    p.win_srows = xrows;
    p.win_dyrows = dyrows;
    p.win_strip_bytes = stage;
    p.M = ntaps * 64;
    p.Ncols = 64;
    p.m_tiles = p.n_tiles = 1;
    p.gN = s->n;
    p.num_kb = (int)((L + kb - 1) / kb);
    // one contiguous range of K-blocks per CTA of a persistent grid
    int splits = grid_size(p.num_kb);
    p.kb_per_split = (p.num_kb + splits - 1) / splits;
    p.zdim = (p.num_kb + p.kb_per_split - 1) / p.kb_per_split;
    pl.ws_main = p.zdim > 1 ? (size_t)p.zdim * p.M * 64 * sizeof(float) : 0;
    return true;
}

// Which tiles run on CTA pairs (see conv_igemm_kernel): 256-column tiles, and the
// 128-column tiles of the weight gradient (its long K-blocks amortise the pair's
// extra synchronisation; the short-K forward and data-gradient passes of 128
// columns measured slower on pairs).  The environment variable DBL_CONV_CTA_PAIRS
// overrides this: 0 = never, 2 = every 128- and 256-column tile.
int cta_pair_level()
{
    static const int level = [] {
        const char* e = getenv("DBL_CONV_CTA_PAIRS");
        return e && (e[0] == '0' || e[0] == '2') ? e[0] - '0' : 1;
    }();
    return level;
}

bool pair_tiles(int BN, bool wgrad)
{
    const int level = cta_pair_level();
    if (level == 0) return false;
    return BN == 256 || (BN == 128 && (wgrad || level == 2));
}

// Window-kernel CTA pairs: 128-column tiles; with DBL_CONV_CTA_PAIRS=2 also the 64-column
// forward pass with resident weights (measured no faster, for comparison); DBL_CONV_CTA_PAIRS=0
// turns them off with the others.
bool win_pairs() { return cta_pair_level() != 0; }

// CTA pairs per tile of the forward pass and the data gradient (conv_splitk_kernel), 256-column pair
// tiles: the count with the least modelled time, in K-blocks (~0.22 us each) of the longest phase.
// One pair per tile runs on the persistent grid, whose epilogues overlap the next tile; split tiles
// pay kTileCost (set-up, first loads, epilogue) every round of the clusters that GB300's 152 SMs hold
// at one time.  A fixed function of the shape: the order of the sums must not depend on the device.
// Measured with 1 / 2 / 4 / 8 pairs (us, data gradient): 36 tiles of 72 K-blocks (3x3x512, batch 512)
// 27.1 / 19.1 / - / -, 16 of 36 (8x8x256, batch 64) 16.7 / 13.3 / 20.8 (two rounds) / -, 10 of 72
// (3x3x512, batch 128) 26.3 / - / 13.8 / -, 6 of 72 (batch 64) 26.2 / - / 13.2 / 12.1.
constexpr int kTileCost = 20;

// Whether the device holds clusters of sk CTA pairs of a split kernel.
template <int BN, int FAM>
bool split_held(int sk)
{
    constexpr int T = SplitCfg<BN, FAM, 2>::THREADS;
    if (sk == 2) return dbl::cluster_held<conv_splitk_kernel<BN, FAM, 2>>(4, T, SplitCfg<BN, FAM, 2>::SMEM);
    if (sk == 4) return dbl::cluster_held<conv_splitk_kernel<BN, FAM, 4>>(8, T, SplitCfg<BN, FAM, 4>::SMEM);
    if constexpr (BN == 256) return dbl::cluster_held<conv_splitk_kernel<BN, FAM, 8>>(16, T, SplitCfg<BN, FAM, 8>::SMEM);
    return false;
}

int fwd_splits(int tiles, int num_kb)
{
    static const int counts[4] = {1, 2, 4, 8}, resident[4] = {76, 36, 15, 7};
    int best = 1;
    int64_t best_cost = INT64_MAX;
    for (int i = 0; i < 4; ++i) {
        const int sk = counts[i];
        if (sk > 1 && (tiles * 2 * sk > kMaxGrid || num_kb < 2 * sk)) continue;
        if (sk > 1 && !split_held<256, kFamFwd>(sk)) break;
        const int64_t rounds = (tiles + resident[i] - 1) / resident[i];
        const int64_t kb = (num_kb + sk - 1) / sk;
        const int64_t cost = sk == 1 ? rounds * kb + kTileCost : rounds * (kb + kTileCost);
        if (cost < best_cost) {
            best_cost = cost;
            best = sk;
        }
    }
    return best;
}

// CTA pairs per tile of the implicit-GEMM weight gradient (conv_splitk_kernel), against `splits` slices of one pair
// each: the least modelled time in SM cycles on a 152-SM GPU.  A K-block takes ~1570 (256 columns) or ~1000
// (128) cycles, a tile ~8000 of set-up, first loads and epilogue, the exchange of partial sums ~2500 of
// barriers and 22 bytes per cycle, the reduce of slices ~5000 and 1800 bytes per cycle.
void wgrad_cluster(Plan& pl, int splits)
{
    static const int counts[3] = {2, 4, 8}, resident[3] = {36, 15, 7};
    ConvParams& p = pl.p;
    const int tiles = p.m_tiles * p.n_tiles;
    const double kbc = pl.BN == 256 ? 1570.0 : 1000.0, acc = 128.0 * pl.BN * 4.0;
    auto reduce = [&](int slices) { return slices > 1 ? 5000.0 + (double)p.M * p.Ncols * 4.0 * slices / 1800.0 : 0.0; };
    double best = ((tiles * splits + 75) / 76) * (double)((p.num_kb + splits - 1) / splits) * kbc + 8000.0 + acc / 40.0 +
                  reduce(splits);
    for (int i = 0; i < 3; ++i) {
        const int sk = counts[i], slices = resident[i] / tiles;
        if (slices < 1 || pl.BN / sk < 32) continue;
        if (!(pl.BN == 256 ? split_held<256, kFamWgrad>(sk) : split_held<128, kFamWgrad>(sk))) break;
        const int kbs = (p.num_kb + slices * sk - 1) / (slices * sk);
        if ((kbs + 1) / 2 > (p.num_kb + splits - 1) / splits) continue;  // an accumulator's K-blocks: no more than a slice's
        const int used = (p.num_kb + kbs * sk - 1) / (kbs * sk);  // no slice without a K-block
        const double cost = kbs * kbc + 10500.0 + acc * (sk - 1) / sk / 22.0 + reduce(used);
        if (cost < best) {
            best = cost;
            pl.sk = sk;
            p.kb_per_split = kbs;
            p.zdim = used;
        }
    }
}

int make_plan(const dbl_conv_shape* s, int pass, Plan& pl)
{
    using dbl::set_error;
    int rc = validate(s, pass == DBL_PASS_FWD ? "conv_fwd" : pass == DBL_PASS_DGRAD ? "conv_dgrad" : "conv_wgrad");
    if (rc) return rc;
    const Geom g = geom(s);
    const int P = out_dim(s->h, s->r, g.sh, g.ph), Q = out_dim(s->w, s->s, g.sw, g.pw);
    ConvParams& p = pl.p;
    memset(&p, 0, sizeof(p));
    const bool c8 = s->c == 8;
    if (!c8 && s->c % 64) return set_error(DBL_ERR_UNSUPPORTED, "conv: input channels must be 8 or a multiple of 64");
    p.ntaps = s->r * s->s;
    p.S = s->s;
    p.Cin = s->c;
    p.zdim = 1;
    if (pass == DBL_PASS_FWD && !c8 && (winpair_setup(s, false, pl) || win_setup(s, s->c, s->k, false, pl))) {
        pl.mode = p.mode = kFwd;
        pl.ws_main = (size_t)kMaxGrid * 2 * s->k * sizeof(float);
    } else if (pass == DBL_PASS_DGRAD && s->c % 64 == 0 && (winpair_setup(s, true, pl) || win_setup(s, s->k, s->c, true, pl))) {
        pl.mode = p.mode = kDgrad;
    } else if (pass == DBL_PASS_WGRAD && (wgrow_setup(s, pl) || wgtap_setup(s, pl) || wgband_setup(s, pl) || wgwin_setup(s, pl))) {
        // conv_wgrow_kernel, conv_wgtap_kernel, conv_wgwin_kernel
    } else if (pass == DBL_PASS_FWD) {
        pl.mode = p.mode = c8 ? kFwdC8 : kFwd;
        if (c8 && p.ntaps > 56) return set_error(DBL_ERR_UNSUPPORTED, "conv_fwd: stem filter too large");
        const int64_t M = (int64_t)s->n * P * Q;
        if (M > INT32_MAX / 2) return set_error(DBL_ERR_UNSUPPORTED, "conv_fwd: too many output pixels");
        p.M = (int)M;
        p.Ncols = s->k;
        pl.BN = c8 ? 64 : choose_bn(s->k);
        pl.cg = !c8 && pair_tiles(pl.BN, false) ? 2 : 1;
        p.m_tiles = (p.M + pl.cg * fwd_tile_rows(pl.BN) - 1) / (pl.cg * fwd_tile_rows(pl.BN));
        p.n_tiles = s->k / pl.BN;
        p.gN = s->n;
        p.gP = P;
        p.gQ = Q;
        p.tstride_h = g.sh;
        p.tstride_w = g.sw;
        p.base_h = -g.ph;
        p.base_w = -g.pw;
        p.cblocks = c8 ? 1 : s->c / 64;
        p.num_kb = c8 ? (p.ntaps + 7) / 8 : p.ntaps * p.cblocks;
        p.ldo = s->k;
        pl.ws_main = (size_t)kMaxGrid * 2 * s->k * sizeof(float);
    } else if (pass == DBL_PASS_DGRAD) {
        if (c8) return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: the 8-channel stem has no data gradient path");
        if (s->r != s->s || g.sh != g.sw || g.ph != g.pw)
            return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: square filters with equal strides and pads only");
        pl.mode = p.mode = kDgrad;
        p.Ncols = s->c;
        pl.BN = choose_bn(s->c);
        p.n_tiles = s->c / pl.BN;
        p.cblocks = s->k / 64;
        p.ldo = s->c;
        p.out_h = s->h;
        p.out_w = s->w;
        p.gN = s->n;
        if (s->stride == 1) {
            if (P != s->h || Q != s->w)
                return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: stride 1 needs 'same' padding (P == H)");
            p.phase_div = 1;
            p.M = s->n * s->h * s->w;
            p.gP = s->h;
            p.gQ = s->w;
            p.base_h = p.base_w = -(s->r - 1 - s->pad);
            int t = 0;
            p.phase_off[0] = 0;
            for (int r2 = 0; r2 < s->r; ++r2)
                for (int s2 = 0; s2 < s->s; ++s2) {
                    if (t >= 16) return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: too many taps");
                    // im2col offset (r2, s2) reads dy at h - (R-1-pad) + r2 = h + pad - r with r = R-1-r2
                    p.tap_oh[t] = (int8_t)r2;
                    p.tap_ow[t] = (int8_t)s2;
                    p.tap_r[t] = (int8_t)(s->r - 1 - r2);
                    p.tap_s[t] = (int8_t)(s->s - 1 - s2);
                    ++t;
                }
            p.phase_off[1] = t;
        } else {
            if ((s->h & 1) || (s->w & 1) || P * 2 != s->h || Q * 2 != s->w)
                return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: stride 2 needs even H, W with P = H/2");
            for (int r = 0; r < s->r; ++r)
                if (r > 1 + s->pad) return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: stride-2 filter too large for pad");
            p.phase_div = 2;
            p.zdim = 4;
            p.gP = s->h / 2;
            p.gQ = s->w / 2;
            p.M = s->n * p.gP * p.gQ;
            p.base_h = p.base_w = 0;
            int t = 0;
            for (int ph = 0; ph < 4; ++ph) {
                const int a = ph >> 1, b = ph & 1;
                p.phase_off[ph] = t;
                for (int r = 0; r < s->r; ++r) {
                    const int dh = a + s->pad - r;
                    if (dh < 0 || (dh & 1)) continue;
                    for (int c2 = 0; c2 < s->s; ++c2) {
                        const int dw = b + s->pad - c2;
                        if (dw < 0 || (dw & 1)) continue;
                        if (t >= 16) return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad: too many taps");
                        p.tap_r[t] = (int8_t)r;
                        p.tap_s[t] = (int8_t)c2;
                        p.tap_oh[t] = (int8_t)(dh / 2);
                        p.tap_ow[t] = (int8_t)(dw / 2);
                        ++t;
                    }
                }
            }
            p.phase_off[4] = t;
        }
        pl.cg = pair_tiles(pl.BN, false) ? 2 : 1;
        p.m_tiles = (p.M + pl.cg * fwd_tile_rows(pl.BN) - 1) / (pl.cg * fwd_tile_rows(pl.BN));
    } else {
        pl.mode = p.mode = c8 ? kWgradC8 : kWgrad;
        p.M = p.ntaps * s->c;  // D rows = (tap, c)
        p.Ncols = s->k;
        pl.BN = c8 ? 64 : choose_bn(s->k);
        pl.cg = !c8 && pair_tiles(pl.BN, true) ? 2 : 1;
        p.m_tiles = c8 ? (p.ntaps + 15) / 16 : (p.M + pl.cg * BM - 1) / (pl.cg * BM);
        p.n_tiles = s->k / pl.BN;
        p.gN = s->n;
        p.gP = P;
        p.gQ = Q;
        p.tstride_h = g.sh;
        p.tstride_w = g.sw;
        p.base_h = -g.ph;
        p.base_w = -g.pw;
        const int64_t pix = (int64_t)s->n * P * Q;
        if ((pix + 127) / 128 > INT32_MAX / 2) return set_error(DBL_ERR_UNSUPPORTED, "conv_wgrad: too many pixels");
        p.num_kb = (int)((pix + 127) / 128);  // K-blocks of 128 output pixels
        const int splits = wgrad_splits(p.m_tiles * p.n_tiles, p.num_kb, p.M, s->k, pl.BN, pl.cg);
        p.kb_per_split = (p.num_kb + splits - 1) / splits;
        p.zdim = splits;
        if (pl.cg == 2) wgrad_cluster(pl, splits);
        pl.ws_main = p.zdim > 1 ? (size_t)p.zdim * p.M * s->k * sizeof(float) : 0;
    }
    p.total_tiles = p.m_tiles * p.n_tiles * p.zdim;
    if (!pl.win && pl.BN == 256 && pl.cg == 2 && (pl.mode == kFwd || pl.mode == kDgrad)) {
        int kb = p.num_kb;  // data gradient: the longest phase
        if (pl.mode == kDgrad)
            for (int z = 0; z < p.zdim; ++z)
                kb = std::max(kb, (p.phase_off[z + 1] - p.phase_off[z]) * p.cblocks);
        pl.sk = fwd_splits(p.total_tiles, kb);
    }
    return DBL_OK;
}

size_t plan_ws(const Plan& pl) { return ((pl.ws_main + 255) / 256) * 256; }

// im2col tensor map over an NHWC tensor.  Bounding-box corners and traversal
// strides are given per spatial axis; the driver takes them innermost axis
// first (W, then H), like the tensor dimensions.
int enc_im2col(CUtensorMap* m, const void* base, int N, int H, int W, int C, int lower_h, int upper_h, int lower_w,
               int upper_w, int stride_h, int stride_w, int channels, int pixels, bool swizzle)
{
    auto fn = dbl::encode_im2col();
    if (!fn) return dbl::set_error(DBL_ERR_CUDA, "conv: cuTensorMapEncodeIm2col unavailable from the driver");
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
    int lo[2] = {lower_w, lower_h}, hi[2] = {upper_w, upper_h};
    cuuint32_t es[4] = {1, (cuuint32_t)stride_w, (cuuint32_t)stride_h, 1};
    CUresult r = fn(m, (dbl::act::kF16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16), 4, const_cast<void*>(base), dims, strides, lo, hi,
                    (cuuint32_t)channels, (cuuint32_t)pixels, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return dbl::set_error(DBL_ERR_CUDA, "conv: im2col tensor map encode failed (%d)", (int)r);
    return DBL_OK;
}

int enc_tiled(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides_bytes,
              const cuuint32_t* box, bool swizzle)
{
    auto fn = dbl::encode_tiled();
    if (!fn) return dbl::set_error(DBL_ERR_CUDA, "conv: cuTensorMapEncodeTiled unavailable from the driver");
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(m, (dbl::act::kF16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16), (cuuint32_t)rank, const_cast<void*>(base), dims,
                    strides_bytes, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return dbl::set_error(DBL_ERR_CUDA, "conv: tiled tensor map encode failed (%d)", (int)r);
    return DBL_OK;
}

template <int BN, int FAM, int CG>
int set_igemm_smem()
{
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(conv_igemm_kernel<BN, FAM, CG>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN, FAM, CG>::SMEM);
        if (e != cudaSuccess) return dbl::cuda_check(e, "conv: set smem attribute");
        attr_set[dev] = true;
    }
    return DBL_OK;
}

// CTA pairs of conv_igemm_kernel<BN, FAM, 2> that fit on the device at once
// (cached per device); at most half the SMs and kMaxGrid / 2.
template <int BN, int FAM>
int resident_pairs()
{
    static int cached[64] = {0};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = -1;
    }
    if (dev >= 0 && dev < 64 && cached[dev] > 0) return cached[dev];
    bool queried = false;  // only a plan the device itself answered for is cached
    int pairs = std::min(dbl::sm_count() / 2, kMaxGrid / 2);
    if (set_igemm_smem<BN, FAM, 2>() == DBL_OK) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(2 * pairs);
        cfg.blockDim = dim3(Cfg<BN, FAM, 2>::THREADS);
        cfg.dynamicSmemBytes = Cfg<BN, FAM, 2>::SMEM;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, conv_igemm_kernel<BN, FAM, 2>, &cfg) == cudaSuccess && n > 0)
        {
            pairs = std::min(pairs, n);
            queried = true;
        } else {
            (void)cudaGetLastError();
        }
    }
    if (pairs < 1) pairs = 1;
    if (queried && dev >= 0 && dev < 64) cached[dev] = pairs;
    return pairs;
}

// Persistent grid of a conv_igemm_kernel plan: one CTA per SM, or one CTA pair
// per two SMs, never more CTAs (pairs) than tiles.
int win_grid(const Plan& pl);

int plan_grid(const Plan& pl)
{
    if (pl.win) return win_grid(pl);
    if (pl.sk > 1) return 2 * pl.sk * pl.p.total_tiles;
    if (pl.cg == 1) return grid_size(pl.p.total_tiles);
    const bool wg = pl.mode == kWgrad || pl.mode == kWgradC8;
    int pairs = pl.BN == 256 ? (wg ? resident_pairs<256, kFamWgrad>() : resident_pairs<256, kFamFwd>())
                             : (wg ? resident_pairs<128, kFamWgrad>() : resident_pairs<128, kFamFwd>());
    if (pairs > pl.p.total_tiles) pairs = pl.p.total_tiles;
    return 2 * std::max(pairs, 1);
}

// Launch attributes of a convolution kernel: a cluster of two (or 2 * SK) for CTA pairs, and, with
// DBL_CONV_PDL=1 in the environment (read once per process), programmatic stream
// serialization, so that the kernel's set-up (barriers, TMEM, descriptor prefetch) overlaps the
// end of the kernel before it (its memory accesses wait in grid_dependency_wait).  Measured on
// GB300: one worker's 224 px step 1.2% faster with it; two workers' iteration on two streams
// 1.1% slower, because CTAs launched early wait on SMs the other stream's kernels need.  Off by
// default.
std::atomic<int> g_conv_pdl_override{-1};  // dbl_set_conv_pdl: -1 = the environment's choice
std::atomic<int> g_conv_stall_next{0};     // dbl_conv_test_stall_next: arms one launch of a kernel that has the hook

bool conv_pdl()
{
    static const bool env_on = [] {
        const char* e = getenv("DBL_CONV_PDL");
        return e && e[0] == '1';
    }();
    const int o = g_conv_pdl_override.load(std::memory_order_relaxed);
    return o < 0 ? env_on : o != 0;
}

int conv_attrs(int cluster, cudaLaunchAttribute (&at)[2])
{
    int n = 0;
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster;
        at[n].val.clusterDim.y = 1;
        at[n].val.clusterDim.z = 1;
        ++n;
    }
    if (conv_pdl()) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    return n;
}

template <int BN, int FAM, int CG>
int launch_cfg(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& a2,
               const CUtensorMap& b2, int grid, cudaStream_t st)
{
    using Cf = Cfg<BN, FAM, CG>;
    int rc = set_igemm_smem<BN, FAM, CG>();
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(Cf::THREADS);
    cfg.dynamicSmemBytes = Cf::SMEM;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = conv_attrs(CG, at);
    ConvParams prm = pl.p;
    if (g_conv_stall_next.exchange(0)) prm.test_stall = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, conv_igemm_kernel<BN, FAM, CG>, a, b, a2, b2, prm);
    if (e != cudaSuccess) {
        dbl::count_launch();
        return dbl::cuda_check(e, "conv_igemm launch");
    }
    return dbl::launch_check("conv_igemm launch");
}

template <int BN, int FAM, int SK>
int launch_splitk(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& a2,
                  const CUtensorMap& b2, int grid, cudaStream_t st)
{
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(conv_splitk_kernel<BN, FAM, SK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             SplitCfg<BN, FAM, SK>::SMEM);
        // a cluster of sixteen CTAs is above the portable size of eight
        if (e == cudaSuccess && 2 * SK > 8)
            e = cudaFuncSetAttribute(conv_splitk_kernel<BN, FAM, SK>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return dbl::cuda_check(e, "conv: set smem attribute");
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(SplitCfg<BN, FAM, SK>::THREADS);
    cfg.dynamicSmemBytes = SplitCfg<BN, FAM, SK>::SMEM;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = conv_attrs(2 * SK, at);
    ConvParams prm = pl.p;
    if (g_conv_stall_next.exchange(0)) prm.test_stall = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, conv_splitk_kernel<BN, FAM, SK>, a, b, a2, b2, prm);
    if (e != cudaSuccess) {
        dbl::count_launch();
        return dbl::cuda_check(e, "conv_splitk launch");
    }
    return dbl::launch_check("conv_splitk launch");
}

// a2, b2: the projection operands of a fused data gradient (unused otherwise).
int launch(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& a2, const CUtensorMap& b2,
           int grid, cudaStream_t st)
{
    const bool wg = pl.mode == kWgrad || pl.mode == kWgradC8;
    if (pl.sk > 1 && wg) {
        if (pl.BN == 256) return pl.sk == 2   ? launch_splitk<256, kFamWgrad, 2>(pl, a, b, a2, b2, grid, st)
                                 : pl.sk == 4 ? launch_splitk<256, kFamWgrad, 4>(pl, a, b, a2, b2, grid, st)
                                              : launch_splitk<256, kFamWgrad, 8>(pl, a, b, a2, b2, grid, st);
        return pl.sk == 2 ? launch_splitk<128, kFamWgrad, 2>(pl, a, b, a2, b2, grid, st)
                          : launch_splitk<128, kFamWgrad, 4>(pl, a, b, a2, b2, grid, st);
    }
    if (pl.sk == 2) return launch_splitk<256, kFamFwd, 2>(pl, a, b, a2, b2, grid, st);
    if (pl.sk == 4) return launch_splitk<256, kFamFwd, 4>(pl, a, b, a2, b2, grid, st);
    if (pl.sk == 8) return launch_splitk<256, kFamFwd, 8>(pl, a, b, a2, b2, grid, st);
    if (pl.cg == 2) {
        if (pl.BN == 256) return wg ? launch_cfg<256, kFamWgrad, 2>(pl, a, b, a2, b2, grid, st)
                                    : launch_cfg<256, kFamFwd, 2>(pl, a, b, a2, b2, grid, st);
        if (pl.BN == 128) return wg ? launch_cfg<128, kFamWgrad, 2>(pl, a, b, a2, b2, grid, st)
                                    : launch_cfg<128, kFamFwd, 2>(pl, a, b, a2, b2, grid, st);
        return dbl::set_error(DBL_ERR_UNSUPPORTED, "conv: CTA pairs need 128 or 256 columns per tile");
    }
    if (wg) {
        if (pl.BN == 256) return launch_cfg<256, kFamWgrad, 1>(pl, a, b, a2, b2, grid, st);
        if (pl.BN == 128) return launch_cfg<128, kFamWgrad, 1>(pl, a, b, a2, b2, grid, st);
        return launch_cfg<64, kFamWgrad, 1>(pl, a, b, a2, b2, grid, st);
    }
    if (pl.BN == 256) return launch_cfg<256, kFamFwd, 1>(pl, a, b, a2, b2, grid, st);
    if (pl.BN == 128) return launch_cfg<128, kFamFwd, 1>(pl, a, b, a2, b2, grid, st);
    return launch_cfg<64, kFamFwd, 1>(pl, a, b, a2, b2, grid, st);
}

template <int BN, bool DG, bool RES, int CG>
int set_win_smem()
{
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(conv_win_kernel<BN, DG, RES, CG>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWinSmemMax);
        if (e != cudaSuccess) return dbl::cuda_check(e, "conv: set smem attribute");
        attr_set[dev] = true;
    }
    return DBL_OK;
}

// CTA pairs of conv_win_kernel<BN, DG, RES, 2> that fit on the device at once with
// `smem` bytes each (one CTA per SM; cached per device), at most half the SMs.
template <int BN, bool DG, bool RES>
int resident_win_pairs(size_t smem)
{
    static int cached[64] = {0};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = -1;
    }
    if (dev >= 0 && dev < 64 && cached[dev] > 0) return cached[dev];
    bool queried = false;  // only a plan the device itself answered for is cached
    int pairs = std::min(dbl::sm_count() / 2, kMaxGrid / 2);
    if (set_win_smem<BN, DG, RES, 2>() == DBL_OK) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(2 * pairs);
        cfg.blockDim = dim3(WinCfg<BN>::THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, conv_win_kernel<BN, DG, RES, 2>, &cfg) == cudaSuccess && n > 0)
        {
            pairs = std::min(pairs, n);
            queried = true;
        } else {
            (void)cudaGetLastError();
        }
    }
    if (pairs < 1) pairs = 1;
    if (queried && dev >= 0 && dev < 64) cached[dev] = pairs;
    return pairs;
}

// Grid of a window-kernel plan: one CTA per SM (never more than tiles), or one CTA
// pair per two SMs (never more pairs than pair units).
int win_grid(const Plan& pl)
{
    if (pl.cg == 1) return grid_size(pl.p.total_tiles);
    const bool dg = pl.mode == kDgrad;
    int pairs = pl.BN == 64 ? resident_win_pairs<64, false, true>(pl.smem)
                : dg        ? resident_win_pairs<128, true, false>(pl.smem)
                            : resident_win_pairs<128, false, false>(pl.smem);
    const int units = (pl.p.total_tiles + 1) / 2;
    if (pairs > units) pairs = units;
    return 2 * std::max(pairs, 1);
}

template <int BN, bool DG, bool RES, int CG>
int launch_win_cfg(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, int grid, cudaStream_t st)
{
    int rc = set_win_smem<BN, DG, RES, CG>();
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(WinCfg<BN>::THREADS);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = conv_attrs(CG, at);
    cudaError_t e = cudaLaunchKernelEx(&cfg, conv_win_kernel<BN, DG, RES, CG>, a, b, pl.p);
    if (e != cudaSuccess) {
        dbl::count_launch();
        return dbl::cuda_check(e, "conv_win launch");
    }
    return dbl::launch_check("conv_win launch");
}

template <bool DG, int CG>
int launch_winpair(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& b32, int grid,
                   cudaStream_t st)
{
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(conv_winpair_kernel<DG, CG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kWinSmemMax);
        if (e != cudaSuccess) return dbl::cuda_check(e, "conv: set smem attribute");
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kWinThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = conv_attrs(CG, at);
    cudaError_t e = cudaLaunchKernelEx(&cfg, conv_winpair_kernel<DG, CG>, a, b, b32, pl.p);
    if (e != cudaSuccess) {
        dbl::count_launch();
        return dbl::cuda_check(e, "conv_winpair launch");
    }
    return dbl::launch_check("conv_winpair launch");
}

// b32: 32-row boxes of the weights (the pixel-pair kernel's CTA pairs).
int launch_win(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& b32, int grid,
               cudaStream_t st)
{
    const bool dg = pl.mode == kDgrad;
    if (pl.winpair)
        return dg           ? launch_winpair<true, 1>(pl, a, b, b32, grid, st)
               : pl.cg == 2 ? launch_winpair<false, 2>(pl, a, b, b32, grid, st)
                            : launch_winpair<false, 1>(pl, a, b, b32, grid, st);
    if (pl.cg == 2) {
        if (pl.BN == 128) return dg ? launch_win_cfg<128, true, false, 2>(pl, a, b, grid, st)
                                    : launch_win_cfg<128, false, false, 2>(pl, a, b, grid, st);
        if (pl.BN == 64 && pl.res && !dg) return launch_win_cfg<64, false, true, 2>(pl, a, b, grid, st);
        return dbl::set_error(DBL_ERR_UNSUPPORTED, "conv: no CTA-pair window kernel for this plan");
    }
    if (pl.BN == 128) return dg ? launch_win_cfg<128, true, false, 1>(pl, a, b, grid, st)
                                : launch_win_cfg<128, false, false, 1>(pl, a, b, grid, st);
    if (pl.res) return dg ? launch_win_cfg<64, true, true, 1>(pl, a, b, grid, st)
                          : launch_win_cfg<64, false, true, 1>(pl, a, b, grid, st);
    return dg ? launch_win_cfg<64, true, false, 1>(pl, a, b, grid, st)
              : launch_win_cfg<64, false, false, 1>(pl, a, b, grid, st);
}

int wgwin_grid(const Plan& pl)
{
    if (pl.wgtap) return pl.p.m_tiles * pl.p.n_tiles * pl.p.zdim * pl.p.win_cl;
    return pl.wgrow || pl.wgband ? pl.p.zdim : grid_size(pl.p.zdim);  // one CTA per slice, whatever the device holds
}

// KERNEL: conv_wgwin_kernel<NACC> or conv_wgrow_kernel (one CTA per split-K range), or
// conv_wgtap_kernel (a CTA per split-K range of each of its tiles).
template <auto KERNEL>
int launch_wgwin(const Plan& pl, const CUtensorMap& a, const CUtensorMap& b, int threads, cudaStream_t st)
{
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWinSmemMax);
        if (e != cudaSuccess) return dbl::cuda_check(e, "conv: set smem attribute");
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cfg.gridDim = dim3(wgwin_grid(pl));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = conv_attrs(pl.wgtap ? pl.p.win_cl : 1, at);
    ConvParams prm = pl.p;
    if (pl.wgtap && g_conv_stall_next.exchange(0)) prm.test_stall = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, KERNEL, a, b, prm);
    if (e != cudaSuccess) {
        dbl::count_launch();
        return dbl::cuda_check(e, "conv_wgwin launch");
    }
    return dbl::launch_check("conv_wgwin launch");
}

// Tensor map of the window kernel's strip operand: one padded row (Wp pixels
// x 64 channels, starting at w = -1) of an NHWC tensor per copy, or `rows` of them of each of `images`.
int enc_win_rows(CUtensorMap* m, const void* base, int N, int H, int W, int C, int Wp, int rows = 1, int images = 1)
{
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t str[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)Wp, (cuuint32_t)rows, (cuuint32_t)images};
    return enc_tiled(m, base, 4, dims, str, box, true);
}

// Tensor map of conv_winpair_kernel's strips: one padded row of one parity per copy, over an NHWC tensor of 64
// channels viewed as [N][H][W/2][2][64].
int enc_winpair_rows(CUtensorMap* m, const void* base, int N, int H, int W, int pitch)
{
    cuuint64_t dims[5] = {64, 2, (cuuint64_t)W / 2, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t str[4] = {128, 256, (cuuint64_t)W * 128, (cuuint64_t)H * W * 128};
    cuuint32_t box[5] = {64, 1, (cuuint32_t)pitch, 1, 1};
    return enc_tiled(m, base, 5, dims, str, box, true);
}

// Rows of one tile of the forward family (see Cfg).
int fwd_tile_rows(int BN) { return BN <= 128 ? 256 : 128; }

// Forward pass.  nparts == nullptr: the channel sums are reduced into ch_sum/ch_sumsq
// (NULL: no statistics).  nparts != nullptr: the per-CTA partials are left in ws
// ([*nparts][2][k]) for the BatchNorm finalize to reduce (dbl_bn_relu_fused_parts).
int conv_fwd_impl(const dbl_conv_shape* s, const void* x, const void* w, void* y, float* ch_sum, float* ch_sumsq,
                  void* ws, size_t ws_bytes, int32_t* nparts, void* stream, const char* who)
{
    using namespace dbl;
    Plan pl;
    int rc = make_plan(s, DBL_PASS_FWD, pl);
    if (rc) return rc;
    if (!x || !w || !y || !aligned16(x) || !aligned16(w) || !aligned16(y))
        return set_error(DBL_ERR_INVALID, "%s: null or misaligned tensor", who);
    if ((ch_sum == nullptr) != (ch_sumsq == nullptr))
        return set_error(DBL_ERR_INVALID, "%s: ch_sum and ch_sumsq go together", who);
    const bool stats = ch_sum != nullptr || nparts != nullptr;
    if (stats && (!ws || ws_bytes < plan_ws(pl)))
        return set_error(DBL_ERR_WORKSPACE, "%s: workspace %zu < %zu bytes", who, ws_bytes, plan_ws(pl));
    CUtensorMap ta, tb, tb32;
    const Geom g = geom(s);
    if (pl.win) {
        if ((rc = pl.winpair ? enc_winpair_rows(&ta, x, s->n, s->h, s->w, pl.p.win_Wp)
                             : enc_win_rows(&ta, x, s->n, s->h, s->w, s->c, pl.p.win_Wp)))
            return rc;
        const int64_t rsc = (int64_t)s->r * s->s * s->c;
        cuuint64_t dims[2] = {(cuuint64_t)rsc, (cuuint64_t)s->k};
        cuuint64_t str[1] = {(cuuint64_t)rsc * 2};
        // a CTA pair stages half the columns each (the pixel-pair kernel: whole taps and half taps)
        cuuint32_t box[2] = {64, (cuuint32_t)(pl.winpair ? 64 : pl.BN / pl.cg)}, box32[2] = {64, 32};
        if ((rc = enc_tiled(&tb, w, 2, dims, str, box, true))) return rc;
        tb32 = tb;
        if (pl.winpair && pl.cg == 2 && (rc = enc_tiled(&tb32, w, 2, dims, str, box32, true))) return rc;
    } else if (pl.mode == kFwdC8) {
        if ((rc = enc_im2col(&ta, x, s->n, s->h, s->w, 8, -g.ph, g.ph - (s->r - 1), -g.pw, g.pw - (s->s - 1), g.sh,
                             g.sw, 8, fwd_tile_rows(pl.BN), false)))
            return rc;
        const int64_t rsc = (int64_t)s->r * s->s * 8;
        cuuint64_t dims[2] = {(cuuint64_t)rsc, (cuuint64_t)s->k};
        cuuint64_t str[1] = {(cuuint64_t)rsc * 2};
        cuuint32_t box[2] = {8, (cuuint32_t)pl.BN};
        if ((rc = enc_tiled(&tb, w, 2, dims, str, box, false))) return rc;
    } else {
        if ((rc = enc_im2col(&ta, x, s->n, s->h, s->w, s->c, -g.ph, g.ph - (s->r - 1), -g.pw, g.pw - (s->s - 1), g.sh,
                             g.sw, 64, fwd_tile_rows(pl.BN), true)))
            return rc;
        const int64_t rsc = (int64_t)s->r * s->s * s->c;
        cuuint64_t dims[2] = {(cuuint64_t)rsc, (cuuint64_t)s->k};
        cuuint64_t str[1] = {(cuuint64_t)rsc * 2};
        cuuint32_t box[2] = {64, (cuuint32_t)(pl.BN / pl.cg)};
        if ((rc = enc_tiled(&tb, w, 2, dims, str, box, true))) return rc;
    }
    pl.p.out = y;
    pl.p.st32 = (reinterpret_cast<uintptr_t>(y) % 32 == 0) && (pl.p.ldo * (int64_t)sizeof(act_t)) % 32 == 0;
    pl.p.stats = stats ? static_cast<float*>(ws) : nullptr;
    const int grid = plan_grid(pl);
    const int parts = pl.sk > 1 ? 2 * pl.p.m_tiles : grid;  // rows of channel-sum partials
    cudaStream_t st = as_stream(stream);
    if ((rc = pl.win ? launch_win(pl, ta, tb, tb32, grid, st) : launch(pl, ta, tb, ta, tb, grid, st))) return rc;
    if (nparts) {
        *nparts = parts;
    } else if (stats) {
        stats_reduce_kernel<<<(s->k + kPartialsChannels - 1) / kPartialsChannels, kPartialsThreads, 0, st>>>(pl.p.stats, parts, s->k, ch_sum, ch_sumsq);
        if ((rc = launch_check("conv stats reduce"))) return rc;
    }
    return DBL_OK;
}


// Data gradient, optionally with the projection shortcut of a ResNet block fused in:
// k2 > 0 adds dgrad of a 1x1 stride-2 pad-0 convolution of the same input (dy2:
// [n, h/2, w/2, k2], w2: [k2][c]) to phase (0,0), the only phase it reaches.
int conv_dgrad_impl(const dbl_conv_shape* s, const void* dy, const void* w, int k2, const void* dy2, const void* w2,
                    void* dx, void* stream, const char* who)
{
    using namespace dbl;
    Plan pl;
    int rc = make_plan(s, DBL_PASS_DGRAD, pl);
    if (rc) return rc;
    if (!dy || !w || !dx || !aligned16(dy) || !aligned16(w) || !aligned16(dx))
        return set_error(DBL_ERR_INVALID, "%s: null or misaligned tensor", who);
    const int P = out_dim(s->h, s->r, s->stride, s->pad), Q = out_dim(s->w, s->s, s->stride, s->pad);
    CUtensorMap ta, tb, ta2, tb2;
    if (pl.win) {
        if ((rc = pl.winpair ? enc_winpair_rows(&ta, dy, s->n, P, Q, pl.p.win_Wp)
                             : enc_win_rows(&ta, dy, s->n, P, Q, s->k, pl.p.win_Wp)))
            return rc;
    } else {
        // im2col over dy [n, P, Q, k]: origins cover the dx grid (stride 1) or one phase grid (stride 2)
        int lower = 0, upper = 0;
        if (s->stride == 1) {
            lower = -(s->r - 1 - s->pad);
            upper = (s->h - 1 + lower) - (P - 1);  // origin range [lower, H-1+lower] against dy's extent P
        }
        if ((rc = enc_im2col(&ta, dy, s->n, P, Q, s->k, lower, upper, lower, upper, 1, 1, 64, fwd_tile_rows(pl.BN),
                             true)))
            return rc;
    }
    // w viewed as [k][r*s][c]: inner c, then tap, then k
    cuuint64_t dims[3] = {(cuuint64_t)s->c, (cuuint64_t)s->r * s->s, (cuuint64_t)s->k};
    cuuint64_t str[2] = {(cuuint64_t)s->c * 2, (cuuint64_t)s->r * s->s * s->c * 2};
    cuuint32_t box[3] = {64, 1, 64};
    if ((rc = enc_tiled(&tb, w, 3, dims, str, box, true))) return rc;
    ta2 = ta;
    tb2 = tb;
    if (k2 > 0) {
        if (pl.win || pl.p.phase_div != 2)
            return set_error(DBL_ERR_UNSUPPORTED, "%s: the projection needs the stride-2 phase path", who);
        // dy2 [n, h/2, w/2, k2] = the phase grid's rows, as [n*P*Q][k2]
        cuuint64_t d2[2] = {(cuuint64_t)k2, (cuuint64_t)s->n * pl.p.gP * pl.p.gQ};
        cuuint64_t s2[1] = {(cuuint64_t)k2 * 2};
        cuuint32_t bx2[2] = {64, (cuuint32_t)fwd_tile_rows(pl.BN)};
        if ((rc = enc_tiled(&ta2, dy2, 2, d2, s2, bx2, true))) return rc;
        // w2 [k2][c] viewed as [k2][1][c], loaded like one tap of w
        cuuint64_t d3[3] = {(cuuint64_t)s->c, 1, (cuuint64_t)k2};
        cuuint64_t s3[2] = {(cuuint64_t)s->c * 2, (cuuint64_t)s->c * 2};
        if ((rc = enc_tiled(&tb2, w2, 3, d3, s3, box, true))) return rc;
        pl.p.proj_kb = k2 / 64;
    }
    pl.p.out = dx;
    pl.p.st32 = (reinterpret_cast<uintptr_t>(dx) % 32 == 0) && (pl.p.ldo * (int64_t)sizeof(act_t)) % 32 == 0;
    const int grid = plan_grid(pl);
    return pl.win ? launch_win(pl, ta, tb, tb, grid, as_stream(stream))
                  : launch(pl, ta, tb, ta2, tb2, grid, as_stream(stream));
}

}  // namespace

extern "C" {

size_t dbl_conv_workspace_bytes(const dbl_conv_shape* shape, int pass)
{
    Plan pl;
    if (pass < 0 || pass > 2 || make_plan(shape, pass, pl) != DBL_OK) return 0;
    return plan_ws(pl);
}

int dbl_conv_plan(const dbl_conv_shape* s, int pass, dbl_conv_plan_info* info)
{
    using namespace dbl;
    if (!info || pass < 0 || pass > 2) return set_error(DBL_ERR_INVALID, "conv_plan: bad arguments");
    Plan pl;
    int rc = make_plan(s, pass, pl);
    if (rc) return rc;
    const bool wgwin = pl.win && pass == DBL_PASS_WGRAD;
    info->kernel = wgwin ? DBL_KERNEL_WINDOW_WGRAD : pl.win ? DBL_KERNEL_WINDOW : DBL_KERNEL_IGEMM;
    info->tile_cols = wgwin && !pl.wgtap ? s->k : pl.BN;
    info->ctas_per_mma = pl.cg;
    info->tiles = pl.p.total_tiles;
    info->zdim = pl.p.zdim;
    info->grid = wgwin ? wgwin_grid(pl) : plan_grid(pl);
    info->smem_bytes = pl.win ? (int64_t)pl.smem : 0;
    return DBL_OK;
}

int dbl_conv_fwd(const dbl_conv_shape* s, const void* x, const void* w, void* y, float* ch_sum, float* ch_sumsq,
                 void* ws, size_t ws_bytes, void* stream)
{
    return conv_fwd_impl(s, x, w, y, ch_sum, ch_sumsq, ws, ws_bytes, nullptr, stream, "conv_fwd");
}

size_t dbl_conv_stats_parts_bytes(const dbl_conv_shape* shape)
{
    Plan pl;
    if (make_plan(shape, DBL_PASS_FWD, pl) != DBL_OK) return 0;
    return (size_t)kMaxGrid * 2 * shape->k * sizeof(float);
}

int dbl_conv_fwd_parts(const dbl_conv_shape* s, const void* x, const void* w, void* y, float* parts,
                       size_t parts_bytes, int32_t* nparts, void* stream)
{
    using dbl::set_error;
    if (!parts || !nparts) return set_error(DBL_ERR_INVALID, "conv_fwd_parts: null partials or count");
    return conv_fwd_impl(s, x, w, y, nullptr, nullptr, parts, parts_bytes, nparts, stream, "conv_fwd_parts");
}

int dbl_conv_dgrad(const dbl_conv_shape* s, const void* dy, const void* w, void* dx, void* ws, size_t ws_bytes,
                   void* stream)
{
    (void)ws;
    (void)ws_bytes;
    return conv_dgrad_impl(s, dy, w, 0, nullptr, nullptr, dx, stream, "conv_dgrad");
}

int dbl_conv_dgrad_proj(const dbl_conv_shape* s, const void* dy, const void* w, int32_t k2, const void* dy2,
                        const void* w2, void* dx, void* ws, size_t ws_bytes, void* stream)
{
    (void)ws;
    (void)ws_bytes;
    using dbl::set_error;
    if (!s) return set_error(DBL_ERR_INVALID, "conv_dgrad_proj: null shape");
    if (s->stride != 2 || (s->stride_w && s->stride_w != 2))
        return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad_proj: the main convolution must have stride 2");
    if (k2 <= 0 || k2 % 64 || k2 > kMaxNcols)
        return set_error(DBL_ERR_UNSUPPORTED, "conv_dgrad_proj: projection channels must be a multiple of 64, <= %d",
                         kMaxNcols);
    if (!dy2 || !w2 || !dbl::aligned16(dy2) || !dbl::aligned16(w2))
        return set_error(DBL_ERR_INVALID, "conv_dgrad_proj: null or misaligned projection tensor");
    return conv_dgrad_impl(s, dy, w, k2, dy2, w2, dx, stream, "conv_dgrad_proj");
}

int dbl_conv_wgrad(const dbl_conv_shape* s, const void* x, const void* dy, float* dw, int accumulate, void* ws,
                   size_t ws_bytes, void* stream)
{
    using namespace dbl;
    Plan pl;
    int rc = make_plan(s, DBL_PASS_WGRAD, pl);
    if (rc) return rc;
    if (!x || !dy || !dw || !aligned16(x) || !aligned16(dy) || !aligned16(dw))
        return set_error(DBL_ERR_INVALID, "conv_wgrad: null or misaligned tensor");
    if (plan_ws(pl) && (!ws || ws_bytes < plan_ws(pl)))
        return set_error(DBL_ERR_WORKSPACE, "conv_wgrad: workspace %zu < %zu bytes", ws_bytes, plan_ws(pl));
    const Geom g = geom(s);
    const int P = out_dim(s->h, s->r, g.sh, g.ph), Q = out_dim(s->w, s->s, g.sw, g.pw);
    CUtensorMap ta, tb;
    cudaStream_t st = as_stream(stream);
    const bool sliced = pl.p.zdim > 1;
    if (pl.win) {
        // rows (and images) per copy
        const int xr = pl.wgrow || pl.wgband || pl.wgtap ? pl.p.win_srows : 1;
        const int yr = pl.wgrow || pl.wgband ? pl.p.win_dyrows : xr, ni = pl.wgtap ? pl.p.win_ni : 1;
        if ((rc = enc_win_rows(&ta, x, s->n, s->h, s->w, s->c, pl.p.win_Wp, xr, ni))) return rc;
        if ((rc = enc_win_rows(&tb, dy, s->n, P, Q, s->k, pl.p.win_Wp, yr, ni))) return rc;
        pl.p.out = sliced ? ws : static_cast<void*>(dw);
        pl.p.wg_accumulate = accumulate;
        if ((rc = pl.wgrow   ? launch_wgwin<conv_wgrow_kernel<false>>(pl, ta, tb, kWinThreads, st)
                  : pl.wgband ? launch_wgwin<conv_wgrow_kernel<true>>(pl, ta, tb, kWinThreads, st)
                  : pl.wgtap ? launch_wgwin<conv_wgtap_kernel>(pl, ta, tb, kWgTapThreads, st)
                  : pl.p.win_R * pl.p.win_S > 4 ? launch_wgwin<conv_wgwin_kernel<5>>(pl, ta, tb, kWinThreads, st)
                                                : launch_wgwin<conv_wgwin_kernel<2>>(pl, ta, tb, kWinThreads, st)))
            return rc;
    } else {
    const bool c8 = pl.mode == kWgradC8;
    if ((rc = enc_im2col(&ta, x, s->n, s->h, s->w, s->c, -g.ph, g.ph - (s->r - 1), -g.pw, g.pw - (s->s - 1), g.sh, g.sw,
                         c8 ? 8 : 64, 128, !c8)))
        return rc;
    cuuint64_t dims[2] = {(cuuint64_t)s->k, (cuuint64_t)s->n * P * Q};
    cuuint64_t str[1] = {(cuuint64_t)s->k * 2};
    cuuint32_t box[2] = {64, 128};
    if ((rc = enc_tiled(&tb, dy, 2, dims, str, box, true))) return rc;
    pl.p.out = sliced ? ws : static_cast<void*>(dw);
    pl.p.wg_accumulate = accumulate;
    if ((rc = launch(pl, ta, tb, ta, tb, plan_grid(pl), st))) return rc;
    }
    if (!sliced) return DBL_OK;
    const int64_t n = (int64_t)pl.p.M * s->k;
    const int lanes = pl.p.zdim > 8 ? 8 : 1;
    int64_t blocks = (n / 4 + 256 / lanes - 1) / (256 / lanes);
    const int64_t cap = (int64_t)sm_count() * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (lanes == 8)
        wgrad_reduce_kernel<8><<<(int)blocks, 256, 0, st>>>(static_cast<const float*>(ws), pl.p.zdim, n, dw, accumulate);
    else
        wgrad_reduce_kernel<1><<<(int)blocks, 256, 0, st>>>(static_cast<const float*>(ws), pl.p.zdim, n, dw, accumulate);
    return launch_check("conv wgrad reduce");
}

int dbl_device_status(int32_t* status)
{
    using namespace dbl;
    if (!status) return set_error(DBL_ERR_INVALID, "device_status: null");
    int rc = cuda_check(cudaDeviceSynchronize(), "device_status sync");
    if (rc) return rc;
    int v = 0, zero = 0;
    if ((rc = cuda_check(cudaMemcpyFromSymbol(&v, g_conv_status, sizeof(int)), "device_status read"))) return rc;
    if ((rc = cuda_check(cudaMemcpyToSymbol(g_conv_status, &zero, sizeof(int)), "device_status clear"))) return rc;
    *status = v;
    return DBL_OK;
}

}  // extern "C"

extern "C" int dbl_conv_test_stall_next(void)
{
    g_conv_stall_next.store(1);
    return DBL_OK;
}

extern "C" int dbl_set_conv_pdl(int32_t mode)
{
    if (mode < -1 || mode > 1) return dbl::set_error(DBL_ERR_INVALID, "set_conv_pdl: mode must be -1, 0 or 1");
    g_conv_pdl_override.store(mode, std::memory_order_relaxed);
    return DBL_OK;
}
