// Learned lane-position proposal: a small BF16 convolutional network on the 4x-downsampled map of
// |G_x w_g| (Eq. 23) ranks the bottom-row starts of Eq. 24-25, and exact energies are evaluated only on
// the best-ranked ones (the exhaustive search of Alg. 7 stays as the fallback).  The paper has no such
// network; the form follows a stated configuration: 3x3 convolutions with 1-16-32-32-16 channels, BF16
// operands with FP32 accumulation, a per-cell logit z (the per-row heatmap is sigmoid(z)), top-k = 32.
//
//   k_conv1     layer 1 (one input channel) from the integer block sums; writes the bf16 input and A1
//   k_conv_tc   layers 2-4 as implicit GEMMs on the tcgen05 tensor cores (bf16 -> f32 in tensor memory):
//               a 16 x 8-cell output tile per MMA (M 128), K = 9 taps x C_in straight from the halo in
//               shared memory; epilogues: bias + ReLU (+ the 1x1 head), or the backward data pass
//               (transposed, flipped weights) times the ReLU mask of the layer below
//   k_wgrad     weight and bias gradients of a layer (mma.sync m16n8k16): M = C_out, N = 9 C_in + 1 (a
//               column of ones gives the bias), K = cells; per-CTA partial sums, then k_wreduce adds them
//               in a fixed order
//   k_loss      head, weighted logistic loss, dz, dS_4 and the head's gradient partials
//   k_adam      Adam (Kingma & Ba, Algorithm 1) on the FP32 master weights, then the bf16 operand copies
//   k_labels    training targets: cells crossed by the Eq. 25 tracks of the selected lanes
//   k_score     coarse-start scores: the heatmap summed along the Eq. 25 track taken in steps of four rows
//   k_topk      the k best coarse starts of a frame -> candidate and evaluated starts
//
// Data layout: cell maps are [n][mh][mw] with mh = ceil(H/4), mw = ceil(W/4); activations are bf16
// [n][mh][mw][C] (channels innermost, 32 or 64 bytes per cell).  Weights: W_l[co][tap][ci] (k = tap C_in
// + ci) for the forward pass and W_l^T[ci][8 - tap][co] for the backward data pass.
#include <cuda_bf16.h>

#include "ld_internal.cuh"
#include "ld_net.cuh"

namespace ld {

namespace {

constexpr int kTileR = 8, kTileC = 16;              // output cells per CTA tile
constexpr int kHaloR = kTileR + 2, kHaloC = kTileC + 2;
constexpr int kConvThreads = 128;                   // 4 warps, two tile rows (two m16 tiles) each
constexpr int kCellThreads = 256;
constexpr float kInScale = 2.384185791015625e-07f;  // 2^-22

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ uint32_t pack_raw(uint16_t lo, uint16_t hi) { return (uint32_t)lo | ((uint32_t)hi << 16); }

__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}

// 32 bytes of a cell at once (a whole sector; the maps' cells are 32 or 64 bytes from a 256-byte aligned base)
__device__ __forceinline__ void ld_cell32(uint32_t (&r)[8], const void *p)
{
    asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p));
}

__device__ __forceinline__ void st_cell32(void *p, const uint32_t (&r)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}

// first cell row a layer must produce for frame f, or INT_MAX when the frame needs nothing
__device__ __forceinline__ int first_needed_row(const FrameState *fs, int f, int depth)
{
    if (!fs)
        return 0;
    const FrameState &s = fs[f];
    if (s.flags & (LD_F_NO_ROAD | LD_F_DEGEN_Y | LD_F_DEGEN_X))
        return 0x7fffffff;
    return (s.v_top >> 2) - depth;
}

// network input of one cell: bf16(f32(sum) 2^-22), as a float
__device__ __forceinline__ float cell_input(int32_t s)
{
    return __bfloat162float(__float2bfloat16_rn(__fmul_rn(__int2float_rn(s), kInScale)));
}

// ---------------------------------------------------------------------------------------------------
// layer 1: one input channel, K = 9, direct FMA per cell
//
// Bound by the cells' instructions (the maps take 10 us): the weights are read four channels at a time and
// multiplied in channel pairs, which halves both.  64 frames of 1242 x 375: 26 us (one weight per load, one
// channel per FMA and 64-bit cell arithmetic: 41 us).
// ---------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kCellThreads) k_conv1(const NetArgs a, const int32_t *xsum, int n,
                                                        const FrameState *fs)
{
    __shared__ __align__(16) float wsm[9 * 16 + 16];   // [tap][co], then the bias
    for (int i = threadIdx.x; i < 16 * 9; i += kCellThreads)
        wsm[(i % 9) * 16 + i / 9] = __bfloat162float(a.wf[0][i]);   // [co][tap]
    for (int i = threadIdx.x; i < 16; i += kCellThreads)
        wsm[144 + i] = a.bias[0][i];
    __syncthreads();
    const uint32_t mh = a.mh, mw = a.mw, cells = n * mh * mw;   // fewer than 2^31: a cell holds over 160 bytes
    for (uint32_t p = blockIdx.x * kCellThreads + threadIdx.x; p < cells; p += gridDim.x * kCellThreads) {
        const uint32_t row = p / mw, f = row / mh;
        const int x = (int)(p - row * mw), y = (int)(row - f * mh);
        if (y < first_needed_row(fs, (int)f, 3))
            continue;
        const int32_t *src = xsum + p;
        float in[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int dy = t / 3 - 1, dx = t % 3 - 1;
            const bool ok = (unsigned)(y + dy) < mh && (unsigned)(x + dx) < mw;
            in[t] = ok ? cell_input(__ldg(src + dy * (int)mw + dx)) : 0.0f;
        }
        if (a.X)
            a.X[p] = __float2bfloat16_rn(in[4]);
        float2 acc[8];   // channel pairs: each half is one correctly rounded fused step, taps in order
#pragma unroll
        for (int c = 0; c < 8; ++c)
            acc[c] = reinterpret_cast<const float2 *>(wsm + 144)[c];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const float2 v = make_float2(in[t], in[t]);
            const float4 *wt = reinterpret_cast<const float4 *>(wsm + t * 16);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 w4 = wt[c];
                acc[2 * c] = __ffma2_rn(make_float2(w4.x, w4.y), v, acc[2 * c]);
                acc[2 * c + 1] = __ffma2_rn(make_float2(w4.z, w4.w), v, acc[2 * c + 1]);
            }
        }
        uint32_t o[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
            o[c] = pack2(fmaxf(acc[c].x, 0.0f), fmaxf(acc[c].y, 0.0f));
        st_cell32(a.act[0] + (size_t)p * 16, o);
    }
}

// ---------------------------------------------------------------------------------------------------
// layers 2-4 (and the backward data pass) on the tensor cores
// ---------------------------------------------------------------------------------------------------
enum Epi { kEpiRelu = 0, kEpiHead = 1, kEpiMask = 2 };

struct ConvIO {
    const __nv_bfloat16 *in;     // [n][mh][mw][CIN]
    const __nv_bfloat16 *wt;     // [COUT][9 CIN]
    const float *bias;           // [COUT] (kEpiRelu, kEpiHead)
    __nv_bfloat16 *out;          // [n][mh][mw][COUT] (kEpiHead: may be null)
    const __nv_bfloat16 *mask;   // [n][mh][mw][COUT] activations whose sign gates the result (kEpiMask)
    const __nv_bfloat16 *wh;     // [16] head weights (kEpiHead)
    const float *bh;             // [1]
    float *z;                    // [n][mh][mw] logits, or the heatmap sigmoid(z) when heat (kEpiHead)
    int n, mh, mw, tiles_r, tiles_c;
    int heat;
    // road rows only (learned detection): frame f needs this layer's output rows >= (v_top >> 2) - depth;
    // tiles entirely above, and frames without a road fit, are skipped (null: every tile)
    const FrameState *fs;
    int depth;
};


// ---------------------------------------------------------------------------------------------------
// layers 2-4 and the backward data pass on the 5th-generation tensor cores (tcgen05, accumulators in
// tensor memory)
//
// Tile: 16 x 8 output cells = the 128 rows (M) of one MMA.  The tile's 18 x 10-cell halo sits in shared
// memory as planes of 8 channels, 16 bytes per cell (plane stride 2880 B, halo row 160 B), which is the
// no-swizzle K-major operand layout for every tap at once: for tap (dy, dx) and 16 input channels the A
// operand starts at the tap's cell of the first plane, its two K halves are one plane apart (leading byte
// offset 2880) and its 16 groups of 8 rows are the tile rows, one halo row apart (stride byte offset 160).
// The weights sit in the matching layout for B (N = C_out rows): per K step of 16 channels, K halves
// C_out x 16 B apart, groups of 8 output channels 128 B apart.  One thread issues the 9 C_in / 16 MMAs of a
// tile (M 128, N C_out, K 16, bf16 -> f32) into one of two accumulators in tensor memory and commits them to
// an mbarrier; meanwhile the CTA reads the other accumulator (tcgen05.ld, one tensor-memory lane quarter per
// warp: a thread gets all C_out channels of one cell) for the previous tile's epilogue and copies the halo of
// the tile after the next in with cp.async (zero-filled outside the map).  Waits are bounded: on a timeout the
// kernel records it in err and stops issuing work.
//
// Bound by latency: a tile's halo, MMAs and epilogue depend on one another, so three halo buffers keep two
// tiles' copies in flight, a warp of its own issues the MMAs (the issuing thread is held up while the queue is
// full and would hold up its warp's epilogue), a warp copies and stores whole cells (32-byte sectors), and the
// mask of the backward pass is fetched before the wait for the MMAs.  64 frames of 1242 x 375, 16->32 / 32->32
// / 32->16 channels: forward 56 / 79 / 83 us, backward 80 / 98 / 75 us (us at the copy bandwidth: 27 / 35 / 27
// and 35 / 53 / 44); with two buffers, no issuing warp and 16-byte pieces 70 / 104 / 98 and 100 / 134 / 115.
// ---------------------------------------------------------------------------------------------------
constexpr int kTcRows = 16, kTcCols = 8;                       // output tile (cells)
constexpr int kTcHR = kTcRows + 2, kTcHC = kTcCols + 2;         // halo
constexpr int kTcPlane = kTcHR * kTcHC * 16;                    // bytes of one 8-channel plane of the halo
constexpr int kTcStages = 3;                                    // halo buffers: one multiplied, two on their way
constexpr int kTcThreads = kConvThreads + 32;                   // copying and epilogue warps, and the issuing one
constexpr unsigned kTcSpin = 1u << 26;                           // wait limit (iterations)

template <int CIN, int COUT>
struct TcSmem {
    static constexpr int halo = (CIN / 8) * kTcPlane;            // one halo buffer
    static constexpr int wts = 9 * CIN * COUT * 2;               // B operand, all taps
    static constexpr size_t bytes = kTcStages * (size_t)halo + wts;
};

__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);   // no swizzle, base offset 0
}

__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t parity)
{
    for (unsigned it = 0; it < kTcSpin; ++it) {
        uint32_t done;
        asm volatile("{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}"
                     : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done)
            return true;
    }
    return false;
}

// (a warp-wide instruction, which callers reach after loops that end per lane: __syncwarp first)
template <int N>
__device__ __forceinline__ void tc_load(uint32_t taddr, uint32_t (&r)[N]);

template <>
__device__ __forceinline__ void tc_load<16>(uint32_t taddr, uint32_t (&r)[16])
{
    __syncwarp();
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

template <>
__device__ __forceinline__ void tc_load<32>(uint32_t taddr, uint32_t (&r)[32])
{
    __syncwarp();
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

template <int CIN, int COUT, int EPI>
__global__ void __launch_bounds__(kTcThreads) k_conv_tc(const ConvIO io, int *err)
{
    using S = TcSmem<CIN, COUT>;
    extern __shared__ __align__(1024) unsigned char tsm_raw[];
    __shared__ uint32_t taddr_s;
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ int stop;                      // a wait ran out: no more MMAs are issued
    unsigned char *wsm = tsm_raw + kTcStages * S::halo;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mh = io.mh, mw = io.mw;
    const int per_frame = io.tiles_r * io.tiles_c, total = io.n * per_frame;
    // weights -> B layout: K step kk = tap (CIN/16) + c16, half h: 16-byte row n at
    // kk (COUT 32) + h (COUT 16) + (n / 8) 128 + (n % 8) 16; a row holds the 8 input channels c16 16 + 8 h ..
    for (int i = tid; i < COUT * 9 * (CIN / 8); i += kTcThreads) {
        const int n = i / (9 * CIN / 8), rem = i % (9 * CIN / 8), tap = rem / (CIN / 8), c8 = rem % (CIN / 8);
        const int kk = tap * (CIN / 16) + (c8 >> 1), h = c8 & 1;
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(io.wt + (size_t)n * 9 * CIN + tap * CIN + c8 * 8));
        *reinterpret_cast<uint4 *>(wsm + kk * COUT * 32 + h * COUT * 16 + (n >> 3) * 128 + (n & 7) * 16) = v;
    }
    const uint32_t mb0 = (uint32_t)__cvta_generic_to_shared(&mbar[0]), mb1 = (uint32_t)__cvta_generic_to_shared(&mbar[1]);
    if (tid == 0) {
        stop = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb0));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb1));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&taddr_s);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(dst));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = taddr_s;
    // the tiles this CTA owns: blockIdx.x, + gridDim.x, ...; those above the road rows are skipped
    auto next_tile = [&](int t) {
        for (; t < total; t += gridDim.x) {
            const int f = t / per_frame, rem = t % per_frame;
            if ((rem / io.tiles_c) * kTcRows + kTcRows - 1 >= first_needed_row(io.fs, f, io.depth))
                return t;
        }
        return total;
    };
    auto load_halo = [&](int t, unsigned char *buf) {
        const int f = t / per_frame, rem = t % per_frame;
        const int y0 = (rem / io.tiles_c) * kTcRows - 1, x0 = (rem % io.tiles_c) * kTcCols - 1;
        for (int i = tid; i < kTcHR * kTcHC * (CIN / 8); i += kConvThreads) {
            const int p = i % (CIN / 8), cell = i / (CIN / 8);   // a warp reads whole cells: full sectors
            const int yy = y0 + cell / kTcHC, xx = x0 + cell % kTcHC;
            const bool in = yy >= 0 && yy < mh && xx >= 0 && xx < mw;
            const __nv_bfloat16 *src = io.in + (((size_t)f * mh + (in ? yy : 0)) * mw + (in ? xx : 0)) * CIN + p * 8;
            cp_async16((uint32_t)__cvta_generic_to_shared(buf + p * kTcPlane + cell * 16), src, in);
        }
    };
    float hw[16], bias[COUT];
    if (EPI == kEpiHead) {
#pragma unroll
        for (int c = 0; c < 16; ++c)
            hw[c] = __bfloat162float(io.wh[c]);
    }
    if (EPI != kEpiMask) {
#pragma unroll
        for (int c = 0; c < COUT; ++c)
            bias[c] = io.bias[c];
    }
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(COUT >> 3) << 17) | ((128u >> 4) << 24);
    const uint32_t wbase = (uint32_t)__cvta_generic_to_shared(wsm);
    bool ok = true;
    const bool issuer = warp == kConvThreads / 32;
    int cur = next_tile(blockIdx.x), nxt = cur < total ? next_tile(cur + gridDim.x) : total, prev = total;
    uint32_t phase[2] = {0u, 0u};
    if (!issuer) {
        if (cur < total)
            load_halo(cur, tsm_raw);
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (nxt < total)
            load_halo(nxt, tsm_raw + S::halo);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int it = 0, st = 0; cur < total || prev < total; ++it) {
        const int b = it & 1;
        if (cur < total) {
            // the halo of `cur` has landed (the next one may be on its way): make it visible to the tensor
            // cores and issue its MMAs
            if (!issuer)
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;");
            if (tid == kConvThreads && !*(volatile int *)&stop) {
                const uint32_t hbase = (uint32_t)__cvta_generic_to_shared(tsm_raw + st * S::halo);
                const uint32_t dacc = tbase + (uint32_t)(b * 32);
#pragma unroll
                for (int tap = 0; tap < 9; ++tap)
#pragma unroll
                    for (int c16 = 0; c16 < CIN / 16; ++c16) {
                        const int kk = tap * (CIN / 16) + c16;
                        const uint64_t ad = tc_desc(hbase + (2 * c16) * kTcPlane + ((tap / 3) * kTcHC + tap % 3) * 16,
                                                    kTcPlane, kTcHC * 16);
                        const uint64_t bd = tc_desc(wbase + kk * COUT * 32, COUT * 16, 128);
                        asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                                     ::"r"(dacc), "l"(ad), "l"(bd), "r"(kIdesc), "r"(kk));
                    }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(b ? mb1 : mb0) : "memory");
            }
        }
        const int nn = nxt < total ? next_tile(nxt + gridDim.x) : total;
        const int pst = st == 0 ? kTcStages - 1 : st - 1;   // the previous tile's buffer
        const int pb = b ^ 1;
        size_t cell = 0;                      // this thread's cell of the previous tile
        bool inside = false;
        uint32_t mk[EPI == kEpiMask ? COUT / 16 : 1][8];
        if (prev < total && !issuer) {
            // the previous tile: its mask is fetched while its MMAs are waited for
            const int f = prev / per_frame, rem = prev % per_frame;
            const int y = (rem / io.tiles_c) * kTcRows + warp * 4 + (lane >> 3), x = (rem % io.tiles_c) * kTcCols + (lane & 7);
            inside = y < mh && x < mw;
            cell = ((size_t)f * mh + y) * mw + x;
            if (EPI == kEpiMask && inside) {
#pragma unroll
                for (int q = 0; q < COUT / 16; ++q)
                    ld_cell32(mk[q], io.mask + cell * COUT + q * 16);
            }
            if (ok && !__all_sync(0xffffffffu, tc_wait(pb ? mb1 : mb0, phase[pb]))) {
                ok = false;   // uniform over the warp (tcgen05.ld is a warp-wide instruction)
                if (lane == 0) {
                    *(volatile int *)&stop = 1;
                    atomicExch(err, 1);
                }
            }
            phase[pb] ^= 1u;
        }
        if (!issuer) {
            // the tile after the next goes into the buffer the previous tile's MMAs have finished with
            if (nn < total && ok)
                load_halo(nn, tsm_raw + pst * S::halo);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        if (prev < total && !issuer) {
            // read the previous tile's accumulator and store its cells
            asm volatile("tcgen05.fence::after_thread_sync;");
            uint32_t r[COUT];
            if (ok)
                tc_load<COUT>(tbase + (uint32_t)(pb * 32) + ((uint32_t)(warp * 32) << 16), r);
            if (ok && inside) {
                if (EPI == kEpiMask) {
#pragma unroll
                    for (int q = 0; q < COUT / 16; ++q) {
                        uint32_t o[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float v0 = bf_lo(mk[q][k]) > 0.0f ? __uint_as_float(r[q * 16 + 2 * k]) : 0.0f;
                            const float v1 = bf_hi(mk[q][k]) > 0.0f ? __uint_as_float(r[q * 16 + 2 * k + 1]) : 0.0f;
                            o[k] = pack2(v0, v1);
                        }
                        st_cell32(io.out + cell * COUT + q * 16, o);
                    }
                } else {
                    float zc = 0.0f;
#pragma unroll
                    for (int q = 0; q < COUT / 16; ++q) {
                        uint32_t o[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const int c = q * 16 + 2 * k;
                            const float v0 = fmaxf(__fadd_rn(__uint_as_float(r[c]), bias[c]), 0.0f);
                            const float v1 = fmaxf(__fadd_rn(__uint_as_float(r[c + 1]), bias[c + 1]), 0.0f);
                            o[k] = pack2(v0, v1);
                            if (EPI == kEpiHead)
                                zc = __fmaf_rn(hw[c + 1], bf_hi(o[k]), __fmaf_rn(hw[c], bf_lo(o[k]), zc));
                        }
                        if (io.out)
                            st_cell32(io.out + cell * COUT + q * 16, o);
                    }
                    if (EPI == kEpiHead) {
                        zc = __fadd_rn(zc, io.bh[0]);
                        io.z[cell] = io.heat ? __frcp_rn(__fadd_rn(1.0f, expf(-zc))) : zc;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
        }
        prev = cur;
        cur = nxt;
        nxt = nn;
        st = st == kTcStages - 1 ? 0 : st + 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tbase));
}

// ---------------------------------------------------------------------------------------------------
// The inference forward in one kernel: layers 1-4 and the head for a 32 x 16-cell output tile, the
// activations kept in shared memory between the layers and the accumulators in tensor memory.
//
// A layer-4 output tile of kFR x kFC cells needs layer 3 on a one-cell border around it, layer 2 on two
// cells, layer 1 on three and the input on four.  Layers 2 and 3 run as 3 x 3 MMA blocks of 16 x 8 cells
// (M 128) over a 48 x 24 region, layer 4 as 2 x 2 blocks; every block is the per-layer kernel's MMA
// sequence (taps in order, then 16-channel K steps, bf16 x bf16 -> f32) on operands in the same plane
// layout (8 channels per plane, 16 bytes per cell; K halves one plane apart, 8-row groups one region row
// apart), so every accumulator, and therefore every activation and logit of the road rows, equals the
// per-layer kernels' bit for bit.  Cells outside the map are stored as zero (the zero padding of the
// next layer); cells a block computes beyond the region the next layer reads are dropped.  One thread
// issues a layer's MMAs into up to nine accumulators (32 tensor-memory columns each) and commits them to
// an mbarrier; the whole CTA waits (bounded), reads the accumulators back (tcgen05.ld, one lane quarter per
// warp, warps w and w + 4 taking the two column halves) and writes the next layer's input.  Layer 1 (one
// input channel) runs on the CUDA cores in the per-layer kernel's operation order.  The next tile's input
// arrives by cp.async while the current tile runs.
//
// Measured on the 64-frame 1242x375 learned detection (top_k 96): 1.26 ms per call against 1.13 ms with one
// kernel per layer.  With about 170 KB of shared memory a CTA is alone on its SM and a tile's phases run
// one after another (issue 21 % active, tensor pipe 12 %), where the per-layer kernels keep four CTAs per
// SM and overlap one tile's MMAs with the next tile's copies; so the per-layer form is the default.
// ---------------------------------------------------------------------------------------------------
constexpr int kFR = 32, kFC = 16;                                // layer-4 output tile (cells)
constexpr int kF1R = kFR + 18, kF1C = kFC + 10;                  // layer-1 region (layer-2 input), origin (-3, -3)
constexpr int kF2R = kF1R, kF2C = kF1C;                          // layer-2 region (layer-3 input), origin (-2, -2)
constexpr int kF3R = kFR + 2, kF3C = kFC + 2;                    // layer-3 region (layer-4 input), origin (-1, -1)
constexpr int kFXR = kF1R + 2, kFXC = kF1C + 2;                  // input region, origin (-4, -4)
constexpr int kFusedThreads = 256;
constexpr int kFP1 = kF1R * kF1C * 16, kFP2 = kF2R * kF2C * 16, kFP3 = kF3R * kF3C * 16;   // plane bytes
constexpr int kFBufA = 2 * kFP1 > 4 * kFP3 ? 2 * kFP1 : 4 * kFP3;                       // layer 1 / layer 3 out
constexpr int kFBufB = 4 * kFP2;                                                         // layer 2 out
constexpr int kFW2 = 9 * 16 * 32 * 2, kFW3 = 9 * 32 * 32 * 2, kFW4 = 9 * 32 * 16 * 2;
constexpr int kFX = kFXR * kFXC * 4;   // one input buffer (raw block sums); two are kept
constexpr size_t kFusedSmem = (size_t)kFBufA + kFBufB + kFW2 + kFW3 + kFW4 + 2 * kFX;
static_assert(kFBufA % 16 == 0 && kFBufB % 16 == 0 && kFX % 16 == 0, "16-byte aligned regions");
// the MMA operands stay inside their regions: block rows x 16 + 15 + 2 and block cols x 8 + 7 + 2
static_assert(2 * 16 + 15 + 2 < kF1R && 2 * 8 + 7 + 2 < kF1C && 16 + 15 + 2 < kF3R && 8 + 7 + 2 < kF3C, "operands in bounds");

struct FusedIO {
    const int32_t *xsum;                 // [n][mh][mw] block sums
    const __nv_bfloat16 *w1;             // [16][9]
    const __nv_bfloat16 *wt[3];          // layers 2-4: [COUT][9 CIN]
    const float *bias[4];
    const __nv_bfloat16 *wh;             // [16]
    const float *bh;                     // [1]
    float *z;                            // [n][mh][mw]
    int n, mh, mw, tiles_r, tiles_c, heat;
    const FrameState *fs;                // road rows only (null: every tile)
};

// weights of one layer -> the B layout of k_conv_tc (per K step kk: K halves COUT x 16 B apart, groups of 8
// output channels 128 B apart)
template <int CIN, int COUT>
__device__ __forceinline__ void fused_load_w(const __nv_bfloat16 *wt, unsigned char *wsm)
{
    for (int i = threadIdx.x; i < COUT * 9 * (CIN / 8); i += kFusedThreads) {
        const int n = i / (9 * CIN / 8), rem = i % (9 * CIN / 8), tap = rem / (CIN / 8), c8 = rem % (CIN / 8);
        const int kk = tap * (CIN / 16) + (c8 >> 1), h = c8 & 1;
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(wt + (size_t)n * 9 * CIN + tap * CIN + c8 * 8));
        *reinterpret_cast<uint4 *>(wsm + kk * COUT * 32 + h * COUT * 16 + (n >> 3) * 128 + (n & 7) * 16) = v;
    }
}

// One thread issues the MMAs of a layer: NBR x NBC blocks of 16 x 8 output cells over an input region of
// RC cells per row (planes of PB bytes), accumulator of block b at column b * COUT.
template <int CIN, int COUT, int NBR, int NBC, int RC, int PB>
__device__ __forceinline__ void fused_mma(uint32_t in_base, uint32_t w_base, uint32_t tbase)
{
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(COUT >> 3) << 17) | ((128u >> 4) << 24);
#pragma unroll 1
    for (int b = 0; b < NBR * NBC; ++b) {
        const int by = b / NBC, bx = b % NBC;
        const uint32_t dacc = tbase + (uint32_t)(b * COUT);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap)
#pragma unroll
            for (int c16 = 0; c16 < CIN / 16; ++c16) {
                const int kk = tap * (CIN / 16) + c16;
                const uint32_t cell = (uint32_t)((by * 16 + tap / 3) * RC + bx * 8 + tap % 3);
                const uint64_t ad = tc_desc(in_base + (uint32_t)(2 * c16 * PB) + cell * 16u, PB, RC * 16);
                const uint64_t bd = tc_desc(w_base + (uint32_t)(kk * COUT * 32), COUT * 16, 128);
                asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                             ::"r"(dacc), "l"(ad), "l"(bd), "r"(kIdesc), "r"(kk));
            }
    }
}

// Epilogue of layer 2 or 3: bias + ReLU -> bf16 into the next layer's input region (ORR x ORC cells,
// planes of PB bytes) whose origin is (oy, ox) in the map; zero outside the map.
template <int NBR, int NBC, int ORR, int ORC, int PB>
__device__ __forceinline__ void fused_epi32(uint32_t tbase, const float *bias, unsigned char *out, int oy, int ox,
                                            int mh, int mw)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, h = warp >> 2;
#pragma unroll 1
    for (int b = 0; b < NBR * NBC; ++b) {
        const int Y = (b / NBC) * 16 + q * 4 + (lane >> 3), X = (b % NBC) * 8 + (lane & 7);
        uint32_t r[16];
        tc_load<16>(tbase + (uint32_t)(b * 32 + 16 * h) + ((uint32_t)(q * 32) << 16), r);
        if (Y < ORR && X < ORC) {
            const int y = oy + Y, x = ox + X;
            const bool in = y >= 0 && y < mh && x >= 0 && x < mw;
#pragma unroll
            for (int pl = 0; pl < 2; ++pl) {
                uint32_t o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = 16 * h + 8 * pl + 2 * k;
                    const float v0 = fmaxf(__fadd_rn(__uint_as_float(r[8 * pl + 2 * k]), bias[c]), 0.0f);
                    const float v1 = fmaxf(__fadd_rn(__uint_as_float(r[8 * pl + 2 * k + 1]), bias[c + 1]), 0.0f);
                    o[k] = in ? pack2(v0, v1) : 0u;
                }
                *reinterpret_cast<uint4 *>(out + (2 * h + pl) * PB + (Y * ORC + X) * 16) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    }
}

// wait for the layer's MMAs (bounded; false on a timeout)
__device__ __forceinline__ bool fused_wait(uint32_t mbar, uint32_t &phase)
{
    const bool ok = tc_wait(mbar, phase);
    phase ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;");
    return ok;
}

__device__ __forceinline__ void fused_sync_for_mma()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic stores -> tensor-core reads
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
}

__global__ void __launch_bounds__(kFusedThreads, 1) k_net_fused(const FusedIO io, int *err)
{
    extern __shared__ __align__(1024) unsigned char fsm[];
    __shared__ uint32_t taddr_s;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ float w1s[16 * 9], b1s[16], b2s[32], b3s[32], b4s[16], hws[16];
    __shared__ int fail_s;
    unsigned char *bufA = fsm, *bufB = fsm + kFBufA;
    unsigned char *w2 = bufB + kFBufB, *w3 = w2 + kFW2, *w4 = w3 + kFW3;
    int32_t *xbuf[2] = {reinterpret_cast<int32_t *>(w4 + kFW4), reinterpret_cast<int32_t *>(w4 + kFW4 + kFX)};
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mh = io.mh, mw = io.mw;
    fused_load_w<16, 32>(io.wt[0], w2);
    fused_load_w<32, 32>(io.wt[1], w3);
    fused_load_w<32, 16>(io.wt[2], w4);
    for (int i = tid; i < 16 * 9; i += kFusedThreads)
        w1s[i] = __bfloat162float(io.w1[i]);
    if (tid < 16) {
        b1s[tid] = io.bias[0][tid];
        b4s[tid] = io.bias[3][tid];
        hws[tid] = __bfloat162float(io.wh[tid]);
    }
    if (tid < 32) {
        b2s[tid] = io.bias[1][tid];
        b3s[tid] = io.bias[2][tid];
    }
    const uint32_t mb = (uint32_t)__cvta_generic_to_shared(&mbar);
    if (tid == 0) {
        fail_s = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&taddr_s);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(dst));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fused_sync_for_mma();   // weights (generic stores) visible to the tensor cores, tensor memory allocated
    const uint32_t tbase = taddr_s;
    const uint32_t aA = (uint32_t)__cvta_generic_to_shared(bufA), aB = (uint32_t)__cvta_generic_to_shared(bufB);
    const uint32_t aw2 = (uint32_t)__cvta_generic_to_shared(w2), aw3 = (uint32_t)__cvta_generic_to_shared(w3),
                   aw4 = (uint32_t)__cvta_generic_to_shared(w4);
    const float bh = io.bh[0];
    uint32_t phase = 0u;
    const int per_frame = io.tiles_r * io.tiles_c, total = io.n * per_frame;
    // the tiles this CTA owns that reach a road row: blockIdx.x, + gridDim.x, ...
    auto next_tile = [&](int t) {
        for (; t < total; t += gridDim.x) {
            const int f = t / per_frame, rem = t % per_frame;
            if ((rem / io.tiles_c) * kFR + kFR - 1 >= first_needed_row(io.fs, f, 0))
                return t;
        }
        return total;
    };
    // the raw block sums of tile t's input region (origin y0 - 4, x0 - 4) into buf by cp.async, zero
    // outside the map
    auto load_x = [&](int t, int32_t *buf) {
        const int f = t / per_frame, rem = t % per_frame;
        const int y0 = (rem / io.tiles_c) * kFR, x0 = (rem % io.tiles_c) * kFC;
        const int32_t *xf = io.xsum + (size_t)f * mh * mw;
        for (int i = tid; i < kFXR * kFXC; i += kFusedThreads) {
            const int y = y0 - 4 + i / kFXC, x = x0 - 4 + i % kFXC;
            const bool in = y >= 0 && y < mh && x >= 0 && x < mw;
            const int32_t *src = xf + (size_t)(in ? y : 0) * mw + (in ? x : 0);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(buf + i)),
                         "l"(src), "r"(in ? 4 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int t = next_tile(blockIdx.x), it = 0;
    if (t < total)
        load_x(t, xbuf[0]);
    for (; t < total; ++it) {
        const int f = t / per_frame, rem = t % per_frame;
        const int y0 = (rem / io.tiles_c) * kFR, x0 = (rem % io.tiles_c) * kFC;
        const int32_t *xs = xbuf[it & 1];
        const int tn = next_tile(t + gridDim.x);
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // this tile's input
        __syncthreads();
        if (tn < total)
            load_x(tn, xbuf[(it + 1) & 1]);   // the next tile's input arrives during this tile
        // layer 1 on the CUDA cores (origin y0 - 3, x0 - 3): the per-layer kernel's FMA order
        for (int i = tid; i < kF1R * kF1C; i += kFusedThreads) {
            const int Y = i / kF1C, X = i % kF1C, y = y0 - 3 + Y, x = x0 - 3 + X;
            float in[9];
#pragma unroll
            for (int tp = 0; tp < 9; ++tp)
                in[tp] = cell_input(xs[(Y + tp / 3) * kFXC + X + tp % 3]);
            const bool inmap = y >= 0 && y < mh && x >= 0 && x < mw;
            uint32_t o[8];
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
                float s0 = b1s[c], s1 = b1s[c + 1];
#pragma unroll
                for (int tp = 0; tp < 9; ++tp) {
                    s0 = __fmaf_rn(w1s[c * 9 + tp], in[tp], s0);
                    s1 = __fmaf_rn(w1s[(c + 1) * 9 + tp], in[tp], s1);
                }
                o[c >> 1] = inmap ? pack2(fmaxf(s0, 0.0f), fmaxf(s1, 0.0f)) : 0u;
            }
            *reinterpret_cast<uint4 *>(bufA + i * 16) = make_uint4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<uint4 *>(bufA + kFP1 + i * 16) = make_uint4(o[4], o[5], o[6], o[7]);
        }
        fused_sync_for_mma();
        // layer 2: 3 x 3 blocks over the layer-1 region -> layer-2 region (origin y0 - 2, x0 - 2)
        if (tid == 0) {
            fused_mma<16, 32, 3, 3, kF1C, kFP1>(aA, aw2, tbase);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb) : "memory");
        }
        if (!fused_wait(mb, phase))
            atomicExch(&fail_s, 1);
        __syncthreads();
        if (fail_s)
            break;
        fused_epi32<3, 3, kF2R, kF2C, kFP2>(tbase, b2s, bufB, y0 - 2, x0 - 2, mh, mw);
        fused_sync_for_mma();
        // layer 3 -> layer-3 region (origin y0 - 1, x0 - 1), into the buffer layer 1 used
        if (tid == 0) {
            fused_mma<32, 32, 3, 3, kF2C, kFP2>(aB, aw3, tbase);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb) : "memory");
        }
        if (!fused_wait(mb, phase))
            atomicExch(&fail_s, 1);
        __syncthreads();
        if (fail_s)
            break;
        fused_epi32<3, 3, kF3R, kF3C, kFP3>(tbase, b3s, bufA, y0 - 1, x0 - 1, mh, mw);
        fused_sync_for_mma();
        // layer 4: 2 x 2 blocks -> bias + ReLU, the 1x1 head, the logit or the heatmap
        if (tid == 0) {
            fused_mma<32, 16, 2, 2, kF3C, kFP3>(aA, aw4, tbase);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb) : "memory");
        }
        if (!fused_wait(mb, phase))
            atomicExch(&fail_s, 1);
        __syncthreads();
        if (fail_s)
            break;
        {
            const int q = warp & 3;
#pragma unroll 1
            for (int b = (warp >> 2) * 2; b < (warp >> 2) * 2 + 2; ++b) {
                const int Y = (b >> 1) * 16 + q * 4 + (lane >> 3), X = (b & 1) * 8 + (lane & 7);
                uint32_t r[16];
                tc_load<16>(tbase + (uint32_t)(b * 16) + ((uint32_t)(q * 32) << 16), r);
                const int y = y0 + Y, x = x0 + X;
                if (y < mh && x < mw) {
                    float zc = 0.0f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int c = 2 * k;
                        const float v0 = fmaxf(__fadd_rn(__uint_as_float(r[c]), b4s[c]), 0.0f);
                        const float v1 = fmaxf(__fadd_rn(__uint_as_float(r[c + 1]), b4s[c + 1]), 0.0f);
                        const uint32_t o = pack2(v0, v1);
                        zc = __fmaf_rn(hws[c + 1], bf_hi(o), __fmaf_rn(hws[c], bf_lo(o), zc));
                    }
                    zc = __fadd_rn(zc, bh);
                    io.z[((size_t)f * mh + y) * mw + x] = io.heat ? __frcp_rn(__fadd_rn(1.0f, expf(-zc))) : zc;
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();   // the next tile overwrites both buffers and the accumulators
        asm volatile("tcgen05.fence::after_thread_sync;");
        t = tn;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (tid == 0 && fail_s)
        atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase));
}

// ---------------------------------------------------------------------------------------------------
// weight gradients: dW[co][tap][ci] = sum_cells dS[co] A[cell + (tap)][ci]; column 9 CIN holds the bias
//
// Per tile of 8 x 16 cells the halo of A and the tile of dS sit in shared memory as the maps have them, a
// cell's channels together, and both MMA operands come out of them with ldmatrix.trans: K is the cells, so
// the transposing load of 8 cells x 8 channels is the fragment, for A at the tap's offset in the halo.
// Cell strides of 2 C + 16 bytes keep the eight 16-byte rows of a matrix on different banks.  The 9 CIN / 16
// groups of 16 columns are spread over the four warps (5 5 4 4 with the bias column on the last one's side,
// or 3 2 2 2); the next tile arrives by cp.async into the other buffer while this one is multiplied.
// kWgradCtasPerSm CTAs of 49 KB share an SM.
// Bound by the tensor pipe's rate for warp-level MMAs (74 of them per 16 cells with 32 x 32 channels; the
// maps would take 35 us at the copy bandwidth).  64 frames of 1242 x 375: 120 / 75 / 80 us for 32x32, 32->16
// and 16->32 channels, and 28 us for the first layer; with B gathered element by element and the dS tile
// transposed by its writers, one buffer, these took 260 / 214 / 176 / 72 us.
// ---------------------------------------------------------------------------------------------------
struct WgradIO {
    const __nv_bfloat16 *dS;     // [n][mh][mw][COUT]
    const __nv_bfloat16 *A;      // [n][mh][mw][CIN]
    float *part;                 // [gridDim.x][COUT][9 CIN + 1]
    int n, mh, mw, tiles_r, tiles_c;
};

template <int CIN, int COUT>
struct WgradShape {
    static constexpr int NCOL = 9 * CIN + 1;
    static constexpr int NG = 9 * CIN / 16;             // groups of 16 columns (two n8 tiles)
    static constexpr int GPW = (NG + 3) / 4;            // per warp, at most
    static constexpr int MT = COUT / 16;
    static constexpr int AS = CIN * 2 + 16;             // cell strides (bytes)
    static constexpr int DS = COUT * 2 + 16;
    static constexpr int abytes = kHaloR * kHaloC * AS, dbytes = kTileR * kTileC * DS;
    static constexpr size_t bytes = 2 * (size_t)(abytes + dbytes);
    static_assert(abytes % 16 == 0 && dbytes % 16 == 0, "16-byte aligned buffers");
};

__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// the dS cells of one tile into shared memory, zero outside the map
template <int COUT>
__device__ __forceinline__ void wgrad_load_ds(const WgradIO &io, int f, int y0, int x0, uint32_t dst)
{
    for (int i = threadIdx.x; i < kTileR * kTileC * (COUT / 8); i += kConvThreads) {
        const int cell = i / (COUT / 8), ch = i % (COUT / 8);
        const int yy = y0 + cell / kTileC, xx = x0 + cell % kTileC;
        const bool in = yy < io.mh && xx < io.mw;
        const size_t c = ((size_t)f * io.mh + (in ? yy : 0)) * io.mw + (in ? xx : 0);
        cp_async16(dst + cell * (COUT * 2 + 16) + ch * 16, io.dS + c * COUT + ch * 8, in);
    }
}

// A fragments (dS^T) of tile row r: matrices (cells 0-7 | 8-15) x (channels 0-7 | 8-15) per 16 channels
template <int MT, int DS>
__device__ __forceinline__ void wgrad_frag_a(uint32_t (&af)[MT][4], uint32_t sd, int r, int lane)
{
    const int cell = r * kTileC + ((lane >> 4) << 3) + (lane & 7);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
        ldsm4_t(af[mt], sd + cell * DS + mt * 32 + ((lane >> 3) & 1) * 16);
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(kConvThreads) k_wgrad(const WgradIO io)
{
    using S = WgradShape<CIN, COUT>;
    extern __shared__ __align__(16) unsigned char gsm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int mh = io.mh, mw = io.mw;
    const int per_frame = io.tiles_r * io.tiles_c;
    const int total = io.n * per_frame;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(gsm);
    // this warp's groups: the first NG % 4 warps have one more
    constexpr int kLess = S::NG / 4, kMore = S::NG % 4;
    const int g0 = warp * kLess + (warp < kMore ? warp : kMore), ng = kLess + (warp < kMore ? 1 : 0);
    const bool has_bias = warp == 3;
    const uint32_t ones = g == 0 ? 0x3f803f80u : 0u;   // the bias tile's only column
    // lane's row of the B matrices: n-tile (lane >> 4), cells (lane >> 3 & 1) * 8 + (lane & 7)
    uint32_t boff[S::GPW];
#pragma unroll
    for (int j = 0; j < S::GPW; ++j) {
        const int col = (g0 + (j < ng ? j : 0)) * 16, tap = col / CIN, ci = col % CIN;
        boff[j] = ((tap / 3) * kHaloC + tap % 3 + ((lane >> 3) & 1) * 8 + (lane & 7)) * S::AS + ci * 2 + (lane >> 4) * 16;
    }
    float acc[S::MT][2 * S::GPW][4], accb[S::MT][4];
#pragma unroll
    for (int mt = 0; mt < S::MT; ++mt) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            accb[mt][q] = 0.0f;
#pragma unroll
        for (int j = 0; j < 2 * S::GPW; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                acc[mt][j][q] = 0.0f;
    }
    auto load_tile = [&](int tile, int buf) {
        const int f = tile / per_frame, rem = tile % per_frame;
        const int y0 = (rem / io.tiles_c) * kTileR, x0 = (rem % io.tiles_c) * kTileC;
        const uint32_t sa = base + buf * (S::abytes + S::dbytes);
        for (int i = tid; i < kHaloR * kHaloC * (CIN / 8); i += kConvThreads) {
            const int cell = i / (CIN / 8), ch = i % (CIN / 8);
            const int yy = y0 - 1 + cell / kHaloC, xx = x0 - 1 + cell % kHaloC;
            const bool in = yy >= 0 && yy < mh && xx >= 0 && xx < mw;
            const size_t c = ((size_t)f * mh + (in ? yy : 0)) * mw + (in ? xx : 0);
            cp_async16(sa + cell * S::AS + ch * 16, io.A + c * CIN + ch * 8, in);
        }
        wgrad_load_ds<COUT>(io, f, y0, x0, sa + S::abytes);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if ((int)blockIdx.x < total)
        load_tile(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // this tile has landed for every thread, and the other buffer is read no more
        if (tile + (int)gridDim.x < total)
            load_tile(tile + gridDim.x, buf ^ 1);
        const uint32_t sa = base + buf * (S::abytes + S::dbytes), sd = sa + S::abytes;
#pragma unroll 2
        for (int r = 0; r < kTileR; ++r) {           // one k16 step per tile row (16 cells)
            uint32_t af[S::MT][4];
            wgrad_frag_a<S::MT, S::DS>(af, sd, r, lane);
#pragma unroll
            for (int j = 0; j < S::GPW; ++j) {
                if (j >= kLess && j >= ng)
                    break;
                uint32_t b[4];
                ldsm4_t(b, sa + r * kHaloC * S::AS + boff[j]);
#pragma unroll
                for (int mt = 0; mt < S::MT; ++mt) {
                    mma16816(acc[mt][2 * j], af[mt][0], af[mt][1], af[mt][2], af[mt][3], b[0], b[1]);
                    mma16816(acc[mt][2 * j + 1], af[mt][0], af[mt][1], af[mt][2], af[mt][3], b[2], b[3]);
                }
            }
            if (has_bias) {
#pragma unroll
                for (int mt = 0; mt < S::MT; ++mt)
                    mma16816(accb[mt], af[mt][0], af[mt][1], af[mt][2], af[mt][3], ones, ones);
            }
        }
    }
    float *part = io.part + (size_t)blockIdx.x * COUT * S::NCOL;
#pragma unroll
    for (int mt = 0; mt < S::MT; ++mt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float *row = part + (mt * 16 + g + (q >> 1) * 8) * S::NCOL;
#pragma unroll
            for (int j = 0; j < 2 * S::GPW; ++j)
                if ((j >> 1) < ng)
                    row[g0 * 16 + j * 8 + 2 * t + (q & 1)] = acc[mt][j][q];
            if (has_bias && t == 0 && (q & 1) == 0)
                row[9 * CIN] = accb[mt][q];
        }
}

// The first layer (one input channel): ten columns (nine taps and the bias) in two n-tiles, so the warps
// split the cells instead, two tile rows each, and their sums are added in warp order at the end.
__global__ void __launch_bounds__(kConvThreads) k_wgrad1(const WgradIO io)
{
    constexpr int COUT = 16, DS = COUT * 2 + 16, kHalo = kHaloR * kHaloC, kPer = (kHalo + kConvThreads - 1) / kConvThreads;
    __shared__ __align__(16) unsigned char sd_raw[2][kTileR * kTileC * DS];
    __shared__ uint16_t sa[2][kHalo];
    __shared__ float red[4][COUT][10];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int mh = io.mh, mw = io.mw, per_frame = io.tiles_r * io.tiles_c, total = io.n * per_frame;
    const uint32_t dbase = (uint32_t)__cvta_generic_to_shared(&sd_raw[0][0]);
    const uint16_t *A = reinterpret_cast<const uint16_t *>(io.A);
    uint16_t next[kPer];
    auto load_tile = [&](int tile, int buf) {
        const int f = tile / per_frame, rem = tile % per_frame;
        const int y0 = (rem / io.tiles_c) * kTileR, x0 = (rem % io.tiles_c) * kTileC;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int i = tid + k * kConvThreads, yy = y0 - 1 + i / kHaloC, xx = x0 - 1 + i % kHaloC;
            next[k] = 0;
            if (i < kHalo && yy >= 0 && yy < mh && xx >= 0 && xx < mw)
                next[k] = __ldg(A + ((size_t)f * mh + yy) * mw + xx);
        }
        wgrad_load_ds<COUT>(io, f, y0, x0, dbase + buf * (kTileR * kTileC * DS));
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[1][2][4] = {};
    const int tapoff = (g / 3) * kHaloC + g % 3;   // tap g, columns 0-7 of the first n-tile
    const uint32_t ones = g == 1 ? 0x3f803f80u : 0u;
    if ((int)blockIdx.x < total)
        load_tile(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, buf ^= 1) {
#pragma unroll
        for (int k = 0; k < kPer; ++k)
            if (tid + k * kConvThreads < kHalo)
                sa[buf][tid + k * kConvThreads] = next[k];
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (tile + (int)gridDim.x < total)
            load_tile(tile + gridDim.x, buf ^ 1);
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const int r = warp * 2 + rr;
            uint32_t af[1][4];
            wgrad_frag_a<1, DS>(af, dbase + buf * (kTileR * kTileC * DS), r, lane);
            const uint16_t *p = &sa[buf][r * kHaloC + tapoff + 2 * t];
            mma16816(acc[0][0], af[0][0], af[0][1], af[0][2], af[0][3], pack_raw(p[0], p[1]), pack_raw(p[8], p[9]));
            // second n-tile: tap 8 (halo offset 2 rows, 2 columns) in column 0, ones in column 1
            const uint16_t *p8 = &sa[buf][(r + 2) * kHaloC + 2 + 2 * t];
            const uint32_t b0 = g == 0 ? pack_raw(p8[0], p8[1]) : ones, b1 = g == 0 ? pack_raw(p8[8], p8[9]) : ones;
            mma16816(acc[0][1], af[0][0], af[0][1], af[0][2], af[0][3], b0, b1);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int co = g + (q >> 1) * 8, c = 2 * t + (q & 1);
        red[warp][co][c] = acc[0][0][q];
        if (c < 2)
            red[warp][co][8 + c] = acc[0][1][q];
    }
    __syncthreads();
    for (int i = tid; i < COUT * 10; i += kConvThreads) {
        const float *r0 = &red[0][0][0] + i;
        io.part[(size_t)blockIdx.x * COUT * 10 + i] =
            __fadd_rn(__fadd_rn(r0[0], r0[COUT * 10]), __fadd_rn(r0[2 * COUT * 10], r0[3 * COUT * 10]));
    }
}

// Sum of nparts partials [nparts][stride] per output, in a fixed order: slice s of a block adds partials
// s, s + slices, ..., then the slices are added by halves.  32 outputs (a 128-byte line of a partial) x 32
// slices per block; the sum is on slice 0's threads.  608 partials: 7-8 us a layer (22 MB for the widest, from
// L2) against 51-56 us with one thread adding all partials of an output one after another; the loss 6 us
// against 22.
constexpr int kRedSlices = 32;

__device__ __forceinline__ float sum_partials(const float *part, int nparts, int stride, int i, bool in)
{
    __shared__ float red[kRedSlices][33];
    const int o = threadIdx.x & 31, sl = threadIdx.x >> 5;
    float s = 0.0f;
    if (in) {
#pragma unroll 4
        for (int k = sl; k < nparts; k += kRedSlices)
            s = __fadd_rn(s, part[(size_t)k * stride + i]);
    }
    red[sl][o] = s;
    for (int h = kRedSlices / 2; h > 0; h >>= 1) {
        __syncthreads();
        if (sl < h)
            red[sl][o] = s = __fadd_rn(s, red[sl + h][o]);
    }
    return s;
}

// The per-CTA partials of a layer, summed and scattered into the flat gradient (layout [co][ci][3][3], b[co]).
__global__ void __launch_bounds__(32 * kRedSlices) k_wreduce(const float *part, int nparts, int cin, int cout,
                                                             float *grad_w, float *grad_b)
{
    const int ncol = 9 * cin + 1;
    const int i = blockIdx.x * 32 + (threadIdx.x & 31);
    const bool in = i < cout * ncol;
    const float s = sum_partials(part, nparts, cout * ncol, i, in);
    if (!in || threadIdx.x >= 32)
        return;
    const int co = i / ncol, col = i % ncol;
    if (col == 9 * cin)
        grad_b[co] = s;
    else
        grad_w[(co * cin + col % cin) * 9 + col / cin] = s;
}

// ---------------------------------------------------------------------------------------------------
// head + loss: z, loss term, dz, dS_4 = bf16(w_h dz [A_4 > 0]); partials (loss, dw_h[16], db_h)
// ---------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kCellThreads) k_loss(const NetArgs a, const uint8_t *labels, int n, float inv_n,
                                                       float pw, float *part)
{
    __shared__ float red[kCellThreads / 32][18];
    const int mh = a.mh, mw = a.mw;
    const long long cells = (long long)n * mh * mw;
    float whv[16];
#pragma unroll
    for (int c = 0; c < 16; ++c)
        whv[c] = __bfloat162float(a.whb[c]);
    const float bh = a.bh[0];
    float acc[18];
#pragma unroll
    for (int k = 0; k < 18; ++k)
        acc[k] = 0.0f;
    for (long long p = blockIdx.x * (long long)kCellThreads + threadIdx.x; p < cells;
         p += (long long)gridDim.x * kCellThreads) {
        uint32_t w32[8];
        ld_cell32(w32, a.act[3] + p * 16);
        float av[16];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            av[2 * k] = bf_lo(w32[k]);
            av[2 * k + 1] = bf_hi(w32[k]);
        }
        float z = 0.0f;
#pragma unroll
        for (int c = 0; c < 16; ++c)
            z = __fmaf_rn(whv[c], av[c], z);
        z = __fadd_rn(z, bh);
        const float y = labels[p] ? 1.0f : 0.0f;
        const float sp = 1.0f / (1.0f + expf(-z));          // sigmoid(z)
        const float sn = 1.0f / (1.0f + expf(z));           // sigmoid(-z)
        const float spz = fmaxf(z, 0.0f) + log1pf(expf(-fabsf(z)));     // softplus(z)
        const float spn = fmaxf(-z, 0.0f) + log1pf(expf(-fabsf(z)));    // softplus(-z)
        acc[0] += pw * y * spn + (1.0f - y) * spz;
        const float dz = ((1.0f - y) * sp - pw * y * sn) * inv_n;
        uint32_t o[8];
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
            const float d0 = av[c] > 0.0f ? whv[c] * dz : 0.0f;
            const float d1 = av[c + 1] > 0.0f ? whv[c + 1] * dz : 0.0f;
            o[c >> 1] = pack2(d0, d1);
            acc[1 + c] = __fmaf_rn(dz, av[c], acc[1 + c]);
            acc[2 + c] = __fmaf_rn(dz, av[c + 1], acc[2 + c]);
        }
        acc[17] += dz;
        st_cell32(a.dS[0] + p * 16, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 18; ++k) {
        float v = acc[k];
        for (int d = 16; d > 0; d >>= 1)
            v += __shfl_down_sync(0xffffffffu, v, d);
        if (lane == 0)
            red[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < 18) {
        float v = 0.0f;
        for (int w = 0; w < kCellThreads / 32; ++w)
            v += red[w][threadIdx.x];
        part[(size_t)blockIdx.x * 18 + threadIdx.x] = v;
    }
}

// loss and the head's gradient from the k_loss partials (fixed order)
__global__ void __launch_bounds__(32 * kRedSlices) k_loss_reduce(const float *part, int nparts, float inv_n,
                                                                 float *grad_head, float *loss_out)
{
    const int k = threadIdx.x & 31;
    const float s = sum_partials(part, nparts, 18, k, k < 18);
    if (k >= 18 || threadIdx.x >= 32)
        return;
    if (k == 0) {
        if (loss_out)
            *loss_out = s * inv_n;
    } else {
        grad_head[k - 1] = s;   // wh[0..15], then bh
    }
}

// ---------------------------------------------------------------------------------------------------
// parameters: Adam step and the bf16 operand copies
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ void store_operand(const NetArgs &a, int i, float v)
{
    // flat layout: per layer W[co][ci][3][3] then b[co]; then wh[16], bh
    int base = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        const int ci_n = net_ch(l), co_n = net_ch(l + 1);
        const int nw = co_n * ci_n * 9;
        if (i < base + nw) {
            const int r = i - base, co = r / (ci_n * 9), ci = (r / 9) % ci_n, tap = r % 9;
            const __nv_bfloat16 b = __float2bfloat16_rn(v);
            a.wf[l][(co * 9 + tap) * ci_n + ci] = b;
            if (l > 0)
                a.wb[l][(ci * 9 + (8 - tap)) * co_n + co] = b;
            return;
        }
        base += nw + co_n;
        if (i < base)
            return;   // bias: read from the master copy
    }
    if (i < base + 16)
        a.whb[i - base] = __float2bfloat16_rn(v);
}

__global__ void k_pack(const NetArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kNetParams)
        store_operand(a, i, a.theta[i]);
}

__global__ void k_adam(const NetArgs a, const float *grad, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kNetParams)
        return;
    const float gi = grad[i];
    const float m = b1 * a.m[i] + (1.0f - b1) * gi;
    const float v = b2 * a.v[i] + (1.0f - b2) * gi * gi;
    a.m[i] = m;
    a.v[i] = v;
    const float th = a.theta[i] - lr * (m / c1) / (sqrtf(v / c2) + eps);   // c1 = 1 - b1^t, c2 = 1 - b2^t
    a.theta[i] = th;
    store_operand(a, i, th);
}

// ---------------------------------------------------------------------------------------------------
// labels, scores, top-k
// ---------------------------------------------------------------------------------------------------
// one thread per (frame, lane): the Eq. 25 track of the lane's start, row by row as in the energy kernel
__global__ void k_labels(const KParams kp, const Work w, const ld_lanes *lanes, uint8_t *labels, int mh, int mw)
{
    const int f = blockIdx.x, l = threadIdx.x;
    if (l >= LD_MAX_LANES)
        return;
    const ld_lanes &L = lanes[f];
    const FrameState &fs = w.fs[f];
    if (l >= L.n_lanes || (fs.flags & (LD_F_NO_ROAD | LD_F_DEGEN_Y | LD_F_DEGEN_X)))
        return;
    const int W = kp.W, H = kp.H, vtop = fs.v_top;
    const float *Vpy = w.rows + (size_t)f * 3 * H + H;
    const float *Vpx = Vpy + H;
    uint8_t *Y = labels + (size_t)f * mh * mw;
    float u = (float)L.start_u[l];
    for (int v = H - 1; v >= vtop; --v) {
        if (v < H - 1) {
            const float vx = Vpx[v + 1], vy = Vpy[v + 1];
            const float num = __fsub_rn(__fadd_rn(vx, __fmul_rn((float)v, u)), __fmul_rn(vy, u));
            const float den = __fsub_rn((float)(v + 1), vy);
            u = __fdiv_rn(num, den);
        }
        const float c = floorf(__fadd_rn(u, 0.5f));
        if (c >= 0.0f && c < (float)W)
            Y[(v >> 2) * mw + ((int)c >> 2)] = 1;
    }
}

// one thread per (frame, coarse start c): the heatmap summed along the track in steps of four rows.  Bound by the
// chain of its steps: the rows' reciprocals are formed once per CTA, and a batch of eight steps is taken before
// the heatmap values of the one before it are added (in row order; a step outside the frame adds 0, which a
// running sum that starts at +0 ignores).  12.6 us for 32 frames of 1242 x 375, 31 us with a division and a
// dependent addition per step.
constexpr int kScThreads = 128, kScBatch = 8;

__global__ void __launch_bounds__(kScThreads) k_score(const KParams kp, const Work w, const float *z, float *scores,
                                                      int mh, int mw)
{
    extern __shared__ float srow[];   // [steps] V_px, V_py, reciprocal of v - V_py, for v = H - 1, H - 5, ...
    const int f = blockIdx.y, c = blockIdx.x * kScThreads + threadIdx.x;
    const int nc = (kp.n_starts + 3) >> 2;
    const FrameState &fs = w.fs[f];
    float acc = 0.0f;
    if (!(fs.flags & LD_F_NO_LANES)) {
        const int W = kp.W, H = kp.H, vtop = fs.v_top;
        const int steps = vtop < H ? (H - 1 - vtop) / 4 + 1 : 0;
        const float *Vpy = w.rows + (size_t)f * 3 * H + H;
        const float *Vpx = Vpy + H;
        const float *zf = z + (size_t)f * mh * mw;
        for (int k = threadIdx.x; k < steps; k += kScThreads) {
            const int v = H - 1 - 4 * k;
            srow[3 * k] = Vpx[v];
            srow[3 * k + 1] = Vpy[v];
            srow[3 * k + 2] = row_reciprocal(__fsub_rn((float)v, Vpy[v]));
        }
        __syncthreads();
        float u = __fadd_rn((float)(4 * c - kp.S0), 1.5f), val[kScBatch] = {};
        for (int k0 = 0; k0 < steps; k0 += kScBatch) {
            int col[kScBatch];
#pragma unroll
            for (int b = 0; b < kScBatch; ++b) {
                const int k = k0 + b;
                col[b] = -1;
                if (k < steps) {
                    col[b] = track_column(u);
                    const float vx = srow[3 * k], vy = srow[3 * k + 1], y = srow[3 * k + 2];
                    const float num = __fmul_rn(4.0f, __fsub_rn(vx, u)), d = __fsub_rn((float)(H - 1 - 4 * k), vy);
                    float q = div_by_row(num, d, y);
                    if (!(fabsf(num) >= kDivNumLo && fabsf(num) <= kDivNumHi && y == y))
                        q = __fdiv_rn(num, d);
                    u = __fadd_rn(u, q);
                }
            }
#pragma unroll
            for (int b = 0; b < kScBatch; ++b) {
                acc = __fadd_rn(acc, val[b]);
                val[b] = (unsigned)col[b] < (unsigned)W ? __ldg(zf + ((H - 1 - 4 * (k0 + b)) >> 2) * mw + (col[b] >> 2)) : 0.0f;
            }
        }
#pragma unroll
        for (int b = 0; b < kScBatch; ++b)
            acc = __fadd_rn(acc, val[b]);
    }
    if (c < nc)
        scores[(size_t)f * nc + c] = acc;
}

// one CTA per frame: the top_k coarse scores (ties to the smaller index), flags of candidate (bit 0) and
// evaluated (bit 1) starts, and the ascending list of evaluated starts
constexpr int kTopThreads = 256;

// order-preserving integer key of a float score (-0 taken as +0, so equal scores give equal keys)
__device__ __forceinline__ uint32_t order_key(float s)
{
    const uint32_t u = __float_as_uint(s == 0.0f ? 0.0f : s);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// sum of v over the threads before this one; red holds kTopThreads / 32 ints
__device__ __forceinline__ int cta_exclusive(int v, int *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d)
            x += y;
    }
    __syncthreads();
    if (lane == 31)
        red[warp] = x;
    __syncthreads();
    int before = 0;
    for (int k = 0; k < warp; ++k)
        before += red[k];
    return before + x - v;
}

__global__ void __launch_bounds__(kTopThreads) k_topk(const KParams kp, const Work w, const float *scores, int top_k,
                                                      uint8_t *cflag, int32_t *elist, int32_t *ecnt, int ecap)
{
    extern __shared__ __align__(16) unsigned char tsm[];
    const int f = blockIdx.x, ns = kp.n_starts, nc = (ns + 3) >> 2;
    uint32_t *key = reinterpret_cast<uint32_t *>(tsm);        // [nc]
    uint8_t *fl = tsm + sizeof(uint32_t) * ((nc + 3) & ~3);   // [ns]
    __shared__ int wsum[kTopThreads / 32];
    __shared__ int red[kTopThreads / 32];
    __shared__ int base;
    __shared__ int hist[256], found[2];
    static_assert(kTopThreads == 256, "a thread clears a bin");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool skip = w.fs[f].flags & LD_F_NO_LANES;
    for (int i = tid; i < nc; i += kTopThreads)
        key[i] = order_key(scores[(size_t)f * nc + i]);
    for (int i = tid; i < ns; i += kTopThreads)
        fl[i] = 0;
    if (tid == 0)
        base = 0;
    __syncthreads();
    if (!skip) {
        // T = the k-th largest key, eight bits at a time from the top: a histogram of the next byte of the keys that
        // agree with T so far, and the highest bin at which the keys from the top reach `need` (four passes of three
        // barriers; bit by bit, 32 counts over the CTA, the kernel took 18 us for 32 frames of 1242 x 375, now 12)
        const int k = top_k < nc ? top_k : nc;
        const int per = (nc + kTopThreads - 1) / kTopThreads;   // contiguous chunks keep index order
        const int c0 = tid * per < nc ? tid * per : nc, c1 = c0 + per < nc ? c0 + per : nc;
        uint32_t T = 0, mask = 0;
        int need = k;                                            // of the keys that agree with T under mask
        for (int shift = 24; shift >= 0; shift -= 8) {
            hist[tid] = 0;
            __syncthreads();
            for (int c = tid; c < nc; c += kTopThreads)
                if ((key[c] & mask) == T)
                    atomicAdd(&hist[(key[c] >> shift) & 255u], 1);
            __syncthreads();
            if (warp == 0) {                                     // lane l: bins 255 - 8 l down to 248 - 8 l
                int sum = 0, incl;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    sum += hist[255 - 8 * lane - j];
                incl = sum;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int o = __shfl_up_sync(0xffffffffu, incl, d);
                    incl += lane >= d ? o : 0;
                }
                const unsigned reach = __ballot_sync(0xffffffffu, incl >= need);   // not empty: k <= nc
                if (lane == __ffs(reach) - 1) {
                    int left = need - (incl - sum), bin = 255 - 8 * lane;
                    while (hist[bin] < left)
                        left -= hist[bin--];
                    found[0] = bin;
                    found[1] = left;
                }
            }
            __syncthreads();
            T |= (uint32_t)found[0] << shift;
            mask |= 255u << shift;
            need = found[1];
        }
        // every key above T is chosen; of the keys equal to T, the first `need` = k - #(key > T) in index order
        int eq = 0;
        for (int c = c0; c < c1; ++c)
            eq += key[c] == T;
        int r = cta_exclusive(eq, red);
        for (int c = c0; c < c1; ++c) {
            bool sel = key[c] > T;
            if (key[c] == T)
                sel = r++ < need;
            if (sel)
                for (int q = 0; q < 4; ++q)
                    if (4 * c + q < ns)
                        fl[4 * c + q] = 1;
        }
    }
    __syncthreads();
    // evaluated = candidate or next to one; per chunk a read phase, then the writes and an ordered compaction
    for (int i0 = 0; i0 < ns; i0 += kTopThreads) {
        const int i = i0 + tid;
        bool ev = false;
        if (i < ns)
            ev = (fl[i] & 1) || (i > 0 && (fl[i - 1] & 1)) || (i + 1 < ns && (fl[i + 1] & 1));
        __syncthreads();
        if (i < ns && ev)
            fl[i] |= 2;
        // ordered compaction of this chunk
        const unsigned bal = __ballot_sync(0xffffffffu, ev);
        if (lane == 0)
            wsum[warp] = __popc(bal);
        __syncthreads();
        int off = base;
        for (int k = 0; k < warp; ++k)
            off += wsum[k];
        off += __popc(bal & ((1u << lane) - 1u));
        if (ev && off < ecap)
            elist[(size_t)f * ecap + off] = i;
        __syncthreads();
        if (tid == 0) {
            int s = 0;
            for (int k = 0; k < kTopThreads / 32; ++k)
                s += wsum[k];
            base += s;
        }
        __syncthreads();
    }
    for (int i = tid; i < ns; i += kTopThreads)
        cflag[(size_t)f * ns + i] = fl[i];
    if (tid == 0)
        ecnt[f] = base < ecap ? base : ecap;
}

}  // namespace

// ---------------------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------------------
// The convolutions, the weight gradients and the fused forward ask for more than the default 48 KB of dynamic shared
// memory (k_conv_tc<32, 32> 53 KB, k_wgrad<32, 32> 49 KB, k_net_fused 173 KB).  The opt-in belongs to the
// current device, so every network makes it for its own (setup_net); the others stay below (k_topk: 2 bytes per start, at
// most 25 KB for the widest frame).

static int grid_for(int tiles, int per_sm)
{
    const int g = sm_count() * per_sm;
    return tiles < g ? tiles : g;
}

__device__ int g_tc_error;   // set when a tensor-core wait ran out (read and cleared by net_tc_status)

template <int CIN, int COUT, int EPI>
static cudaError_t conv(ConvIO io, cudaStream_t s)
{
    using S = TcSmem<CIN, COUT>;
    io.tiles_r = (io.mh + kTcRows - 1) / kTcRows;
    io.tiles_c = (io.mw + kTcCols - 1) / kTcCols;
    int *err = nullptr;
    cudaError_t e = cudaGetSymbolAddress((void **)&err, g_tc_error);
    if (e != cudaSuccess)
        return e;
    const int tiles = io.n * io.tiles_r * io.tiles_c;
    k_conv_tc<CIN, COUT, EPI><<<grid_for(tiles, 4), kTcThreads, S::bytes, s>>>(io, err);
    return cudaGetLastError();
}

static cudaError_t net_forward_fused(const NetArgs &a, const int32_t *xsum, int n, float *z, bool heat, cudaStream_t s,
                                     const FrameState *road)
{
    FusedIO io{};
    io.xsum = xsum;
    io.w1 = a.wf[0];
    for (int l = 0; l < 3; ++l)
        io.wt[l] = a.wf[l + 1];
    for (int l = 0; l < 4; ++l)
        io.bias[l] = a.bias[l];
    io.wh = a.whb;
    io.bh = a.bh;
    io.z = z;
    io.n = n;
    io.mh = a.mh;
    io.mw = a.mw;
    io.tiles_r = (a.mh + kFR - 1) / kFR;
    io.tiles_c = (a.mw + kFC - 1) / kFC;
    io.heat = heat ? 1 : 0;
    io.fs = road;
    int *err = nullptr;
    cudaError_t e = cudaGetSymbolAddress((void **)&err, g_tc_error);
    if (e != cudaSuccess)
        return e;
    k_net_fused<<<grid_for(n * io.tiles_r * io.tiles_c, 1), kFusedThreads, kFusedSmem, s>>>(io, err);
    return cudaGetLastError();
}

// Shared-memory opt-ins of the current device (each always to the same value: networks share the kernels).
cudaError_t setup_net()
{
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto *kernel, size_t bytes) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    allow(k_conv_tc<16, 32, kEpiRelu>, TcSmem<16, 32>::bytes);
    allow(k_conv_tc<32, 32, kEpiRelu>, TcSmem<32, 32>::bytes);
    allow(k_conv_tc<32, 16, kEpiHead>, TcSmem<32, 16>::bytes);
    allow(k_conv_tc<16, 32, kEpiMask>, TcSmem<16, 32>::bytes);
    allow(k_conv_tc<32, 32, kEpiMask>, TcSmem<32, 32>::bytes);
    allow(k_conv_tc<32, 16, kEpiMask>, TcSmem<32, 16>::bytes);
    allow(k_wgrad<32, 16>, WgradShape<32, 16>::bytes);
    allow(k_wgrad<32, 32>, WgradShape<32, 32>::bytes);
    allow(k_wgrad<16, 32>, WgradShape<16, 32>::bytes);
    allow(k_net_fused, kFusedSmem);
    return e;
}

cudaError_t net_forward(const NetArgs &a, const int32_t *xsum, int n, float *z, bool keep_a4, bool heat,
                        cudaStream_t s, const FrameState *road)
{
    if (!keep_a4 && a.fused)   // inference in one kernel, the activations never leave the SM
        return net_forward_fused(a, xsum, n, z, heat, s, road);
    const long long cells = (long long)n * a.mh * a.mw;
    const int g1 = (int)((cells + kCellThreads - 1) / kCellThreads);
    k_conv1<<<grid_for(g1, 8), kCellThreads, 0, s>>>(a, xsum, n, road);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    ConvIO io{};
    io.n = n;
    io.mh = a.mh;
    io.mw = a.mw;
    io.tiles_r = (a.mh + kTileR - 1) / kTileR;
    io.tiles_c = (a.mw + kTileC - 1) / kTileC;
    io.fs = road;
    io.in = a.act[0];
    io.wt = a.wf[1];
    io.bias = a.bias[1];
    io.out = a.act[1];
    io.depth = 2;
    if ((e = conv<16, 32, kEpiRelu>(io, s)) != cudaSuccess)
        return e;
    io.in = a.act[1];
    io.wt = a.wf[2];
    io.bias = a.bias[2];
    io.out = a.act[2];
    io.depth = 1;
    if ((e = conv<32, 32, kEpiRelu>(io, s)) != cudaSuccess)
        return e;
    io.depth = 0;
    io.in = a.act[2];
    io.wt = a.wf[3];
    io.bias = a.bias[3];
    io.out = keep_a4 ? a.act[3] : nullptr;
    io.wh = a.whb;
    io.bh = a.bh;
    io.z = z;
    io.heat = heat ? 1 : 0;
    return conv<32, 16, kEpiHead>(io, s);
}

template <int CIN, int COUT>
static cudaError_t wgrad(const NetArgs &a, const __nv_bfloat16 *dS, const __nv_bfloat16 *A, int n, float *gw,
                         float *gb, cudaStream_t s)
{
    WgradIO io{};
    io.dS = dS;
    io.A = A;
    io.part = a.part;
    io.n = n;
    io.mh = a.mh;
    io.mw = a.mw;
    io.tiles_r = (a.mh + kTileR - 1) / kTileR;
    io.tiles_c = (a.mw + kTileC - 1) / kTileC;
    const int G = grid_for(n * io.tiles_r * io.tiles_c, kWgradCtasPerSm);
    if constexpr (CIN == 1) {
        static_assert(COUT == 16, "k_wgrad1 is the first layer's");
        k_wgrad1<<<G, kConvThreads, 0, s>>>(io);
    } else {
        k_wgrad<CIN, COUT><<<G, kConvThreads, WgradShape<CIN, COUT>::bytes, s>>>(io);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    const int outs = COUT * (9 * CIN + 1);
    k_wreduce<<<(outs + 31) / 32, 32 * kRedSlices, 0, s>>>(a.part, G, CIN, COUT, gw, gb);
    return cudaGetLastError();
}

cudaError_t net_backward(const NetArgs &a, const uint8_t *labels, int n, float pw, float *grad, float *loss,
                         cudaStream_t s)
{
    const long long cells = (long long)n * a.mh * a.mw;
    const float inv_n = 1.0f / (float)cells;
    const int gl = (int)((cells + kCellThreads - 1) / kCellThreads);
    const int GL = grid_for(gl, 4);
    k_loss<<<GL, kCellThreads, 0, s>>>(a, labels, n, inv_n, pw, a.part_head);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    k_loss_reduce<<<1, 32 * kRedSlices, 0, s>>>(a.part_head, GL, inv_n, grad + kNetParams - 17, loss);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    // parameter offsets
    int off[4], cur = 0;
    for (int l = 0; l < 4; ++l) {
        off[l] = cur;
        cur += net_ch(l + 1) * net_ch(l) * 9 + net_ch(l + 1);
    }
    auto gw = [&](int l) { return grad + off[l]; };
    auto gb = [&](int l) { return grad + off[l] + net_ch(l + 1) * net_ch(l) * 9; };
    ConvIO io{};
    io.n = n;
    io.mh = a.mh;
    io.mw = a.mw;
    io.tiles_r = (a.mh + kTileR - 1) / kTileR;
    io.tiles_c = (a.mw + kTileC - 1) / kTileC;
    // layer 4: dS_4 in dS[0] (16 channels), A_3 (32)
    if ((e = wgrad<32, 16>(a, a.dS[0], a.act[2], n, gw(3), gb(3), s)) != cudaSuccess)
        return e;
    io.in = a.dS[0];
    io.wt = a.wb[3];
    io.mask = a.act[2];
    io.out = a.dS[1];
    if ((e = conv<16, 32, kEpiMask>(io, s)) != cudaSuccess)    // dS_3 (32)
        return e;
    if ((e = wgrad<32, 32>(a, a.dS[1], a.act[1], n, gw(2), gb(2), s)) != cudaSuccess)
        return e;
    io.in = a.dS[1];
    io.wt = a.wb[2];
    io.mask = a.act[1];
    io.out = a.dS[0];
    if ((e = conv<32, 32, kEpiMask>(io, s)) != cudaSuccess)    // dS_2 (32)
        return e;
    if ((e = wgrad<16, 32>(a, a.dS[0], a.act[0], n, gw(1), gb(1), s)) != cudaSuccess)
        return e;
    io.in = a.dS[0];
    io.wt = a.wb[1];
    io.mask = a.act[0];
    io.out = a.dS[1];
    if ((e = conv<32, 16, kEpiMask>(io, s)) != cudaSuccess)    // dS_1 (16)
        return e;
    return wgrad<1, 16>(a, a.dS[1], a.X, n, gw(0), gb(0), s);
}

int net_tc_status()
{
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int)) != cudaSuccess)
        return -1;
    if (v)
        cudaMemcpyToSymbol(g_tc_error, &zero, sizeof(int));
    return v;
}

cudaError_t net_pack(const NetArgs &a, cudaStream_t s)
{
    k_pack<<<(kNetParams + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t net_adam(const NetArgs &a, const float *grad, float lr, float b1, float b2, float eps, float c1, float c2,
                     cudaStream_t s)
{
    k_adam<<<(kNetParams + 255) / 256, 256, 0, s>>>(a, grad, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t net_labels(const KParams &kp, const Work &w, const ld_lanes *lanes, uint8_t *labels, int mh, int mw,
                       cudaStream_t s)
{
    k_labels<<<kp.n_frames, 32, 0, s>>>(kp, w, lanes, labels, mh, mw);
    return cudaGetLastError();
}

cudaError_t net_propose(const KParams &kp, const Work &w, const float *z, int mh, int mw, int top_k, float *scores,
                        uint8_t *cflag, int32_t *elist, int32_t *ecnt, int ecap, cudaStream_t s)
{
    const int nc = (kp.n_starts + 3) >> 2;
    dim3 g1((nc + kScThreads - 1) / kScThreads, kp.n_frames);
    k_score<<<g1, kScThreads, sizeof(float) * 3 * (size_t)((kp.H + 3) / 4), s>>>(kp, w, z, scores, mh, mw);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    const size_t smem = sizeof(float) * (size_t)((nc + 3) & ~3) + (size_t)kp.n_starts;
    k_topk<<<kp.n_frames, kTopThreads, smem, s>>>(kp, w, scores, top_k, cflag, elist, ecnt, ecap);
    return cudaGetLastError();
}

}  // namespace ld
