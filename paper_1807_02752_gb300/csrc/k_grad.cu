// Sec. 2.3.1: road mask, bilateral filter (Eq. 15-16), Sobel gradients, edge test and sparse V_px votes
// (Eq. 17), for the road rows of every frame.
//
// One CTA owns a tile of R rows x 64 four-pixel groups (256 columns) of one frame: the road test, the edge
// test and the votes of those pixels.  It stages the image region its stencils reach in shared memory as
// 2 I, with a sentinel value outside the frame whose range weight is 0 (this is the clipped window of
// Eq. 15).  Small tiles keep a CTA at about 50 KB of shared memory, so four run on an SM and one CTA's
// barriers and loads overlap the others' arithmetic.
//
// Exact pruning: a road pixel whose neighbourhood is provably too flat to pass the edge test (an image
// range of at most kp.flat_range over the windows of its 3x3 neighbours; the bound is derived and
// computed on the host, flat_range() in ld_api.cu) leaves the road mask.  On the 1242x375 workload about
// three quarters of the bilateral work goes with those pixels, and every edge, G and vote stays as the
// full computation gives them.
//
// The bilateral output is computed only at the pixel pairs holding a pixel of the 3x3 neighbourhood of a
// remaining road pixel of the tile (neighbouring tiles compute their shared border pairs each).  Weights
// are Q15 integers, w = (ws * wr[|I(i,j) - I(u,v)|] + 2^14) >> 15, sums are exact, and the output is
// (2 sum(w I) + sum(w)) / (2 sum(w)), so the result does not depend on the order of the taps.
//
// GB300 mapping of the bilateral:
//   - taps at equal distance share ws and the range weight depends on |I(i,j) - I(u,v)| only, so w depends
//     on (distance class, |dI|); the CTA builds one 512-entry uint16 table per class in shared memory and
//     a tap costs one absolute-difference-add (__usad), one table load and two 32-bit accumulations
//     (sum(w) and sum(w 2 I)).  Indexing by |dI| keeps the common small differences in half of the banks;
//   - the tile stores 2 I (a byte offset into a table), so the table address is base_c + |2 I(i,j) - 2 I(u,v)|
//     with a compile-time class offset; the sentinel 2 x 511 outside the frame lands in the zero half of
//     every table;
//   - a thread filters 2 horizontally adjacent pixels, sharing each window row it loads.
//
// Bound by instruction issue and the shared-memory pipe together (issue slots 60 % busy, shared-memory wavefronts
// 56 %, ALU 50 %); the frames themselves are 22 us at the copy bandwidth for 64 of 1242 x 375.  Four CTAs of 256
// threads per SM measured best (rows 8 / 12 / 20 / 24 a CTA, 384 and 512 threads, five CTAs of 12 rows: all slower).
// The row tiles are launched from the bottom of the frames up: the top ones hold little road and fill the last wave.
// 64 frames: 240 us, sixteen of 1920 x 1080: 320 us, one frame of 1242 x 375: 27 us.  With groups of four pixels
// filtered whole by fully unrolled code, byte loads of the image, a flatness test that took the windows' ranges
// horizontally first, and division, atomics and stores under each group's own branches: 297 / 365 / 31 us.
//
// Each remaining road pixel with G_x^2 + G_y^2 > thr^2 is an edge pixel.  Its vote column is
// floor(u + (v - V_py(v)) G_y / G_x + 0.5) in float32 (the line through the pixel perpendicular to the
// gradient meets row V_py there), kept when inside [0, W).  Edge pixels and votes are appended to per-row
// lists through one global atomic per row and tile (order within a row is arbitrary; every consumer sums
// over them); k_vdisp zeroes the per-row counts.
#include "ld_internal.cuh"

namespace ld {

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kGroups = 64;                // four-pixel groups per CTA (256 columns)
constexpr int kTabEntries = 512;           // T_c[|dI|]: |dI| <= 255, zero from 256 on (where the sentinel lands)
constexpr int kTabBytes = kTabEntries * 2;  // one uint16 table per distance class

// Distance class of every tap (rank of dx^2 + dy^2 among the distinct values of the window), as byte
// offsets of the class tables; a compile-time table, so an unrolled tap loop folds them into the loads.
template <int RHO>
__host__ __device__ constexpr int cls_rank(int d2)
{
    int r = 0;
    for (int s = 0; s < d2; ++s) {
        bool seen = false;
        for (int dy = 0; dy <= RHO; ++dy)
            for (int dx = 0; dx <= RHO; ++dx)
                if (dx * dx + dy * dy == s)
                    seen = true;
        r += seen ? 1 : 0;
    }
    return r;
}
template <int RHO>
struct ClsOffsets {
    int v[(2 * RHO + 1) * (2 * RHO + 1)];
};
template <int RHO>
__host__ __device__ constexpr ClsOffsets<RHO> make_cls_offsets()
{
    ClsOffsets<RHO> o{};
    for (int dy = 0; dy <= 2 * RHO; ++dy)
        for (int dx = 0; dx <= 2 * RHO; ++dx)
            o.v[dy * (2 * RHO + 1) + dx] = cls_rank<RHO>((dy - RHO) * (dy - RHO) + (dx - RHO) * (dx - RHO)) * kTabBytes;
    return o;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t lds_u16(uint32_t addr)
{
    uint16_t v;
    asm("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}

// Bilateral output of 2 pixels whose windows start at tile row br and tile column u0, an even one (the pixels sit
// at tile row br + RHO, columns u0 + RHO ..); nv of them lie inside the frame.  The tile holds 2 I with the
// sentinel outside the frame.
// sum(w) <= 121 * 2^15 and sum(w 2 I) <= 121 * 2^15 * 510 < 2^31 both fit 32-bit accumulators (one 64-bit
// accumulator for both, a wide multiply-add per tap, is slower: 250 us against 240 for the 64-frame call).
// The rows at the same distance above and below the pixels share their class offsets and are one piece of code, and
// a thread has two pixels: unrolled over all rows of four pixels the taps are 31 KB of code, and every eighth
// stalled warp waited for instructions.  (Two lanes a pair, one for the rows above and one for those below, fill
// the last warps better but pay more for loads: 252 us.)
template <int RHO>
__device__ __forceinline__ uint32_t bilateral2(const uint16_t *tile, int TWP, int br, int u0, int nv, uint32_t tab)
{
    constexpr int N = 2 * RHO + 1;
    constexpr ClsOffsets<RHO> kOff = make_cls_offsets<RHO>();
    const uint16_t *crow = tile + (size_t)(br + RHO) * TWP + u0;
    uint32_t base[2], sw[2] = {0u, 0u}, swi[2] = {0u, 0u};
#pragma unroll
    for (int p = 0; p < 2; ++p)
        base[p] = p < nv ? crow[RHO + p] : 0u;  // pixels past the right edge: any valid index
#pragma unroll
    for (int ady = 0; ady <= RHO; ++ady) {
#pragma unroll 1
        for (int sg = -1; sg <= (ady ? 1 : -1); sg += 2) {
            const uint32_t *rowp = reinterpret_cast<const uint32_t *>(crow + sg * ady * TWP);
            uint32_t q[2 * RHO + 2];
#pragma unroll
            for (int l = 0; l <= RHO; ++l) {
                const uint32_t v = rowp[l];
                q[2 * l] = v & 0xffffu;
                q[2 * l + 1] = v >> 16;
            }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
#pragma unroll
                for (int dx = 0; dx < N; ++dx) {
                    const uint32_t qq = q[p + dx];
                    const uint32_t wq = lds_u16(__usad(qq, base[p], tab) + (uint32_t)kOff.v[(RHO + ady) * N + dx]);
                    sw[p] += wq;
                    swi[p] += wq * qq;
                }
            }
        }
    }
    uint32_t out = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const uint32_t b = sw[p] ? (swi[p] + sw[p]) / (2u * sw[p]) : 0u;  // (2 sum(wI) + sum(w)) / (2 sum(w))
        out |= (b & 0xffu) << (8 * p);
    }
    return out;
}

// Four-column blocks of a group's test window: frame columns 4g - RHO - 4 .. 4g + RHO + 5 at least.
template <int RHO>
constexpr int kFlatBlocks = (2 * RHO + 10 + 3) / 4;
constexpr int kFlatRows = 8;               // rows of ranges a thread of the flatness test forms

// Shared-memory layout of a tile (bytes; every region 16-byte aligned).
struct GradTile {
    int TWP, TR, nj, IWO, IWB, NGB, NB;
    size_t o_tab, o_tile, o_live, o_ibf, o_gl, o_row, o_need, bytes;
};
template <int RHO>
__host__ __device__ inline GradTile grad_tile(int nr, int nj, int n_cls)
{
    GradTile t;
    t.nj = nj;
    t.TWP = (4 * nj + 2 * RHO + 8 + 3) & ~3;  // tile columns: frame columns 4 j0 - RHO - 4 ..
    t.TR = nr + 2 * RHO + 2;                  // tile rows: frame rows r0 - RHO - 1 ..
    t.IWO = 4 * nj;                           // owned pixels per row
    t.NGB = nj + 2;                           // bilateral groups per row: j0 - 1 .. j0 + nj
    t.IWB = 4 * t.NGB;
    size_t o = 0;
    auto take = [&](size_t b) {
        const size_t r = o;
        o = (o + b + 15) & ~(size_t)15;
        return r;
    };
    t.o_tab = take((size_t)kTabBytes * n_cls);
    // the image tile; once filtered, the edge lists of the rows the warps work on
    const size_t tile = 2 * (size_t)t.TR * t.TWP, lists = sizeof(short4) * (size_t)(nr < kWarps ? nr : kWarps) * t.IWO;
    t.o_tile = take(tile > lists ? tile : lists);
    t.o_live = take((size_t)nr * t.IWO);
    // the bilateral output; before it, the ranges of the flatness test
    t.NB = nj + kFlatBlocks<RHO> - 1;
    const size_t ibf = (size_t)(nr + 2) * t.IWB, ranges = 4 * (size_t)nr * t.NB;
    t.o_ibf = take(ibf > ranges ? ibf : ranges);
    t.o_gl = take(2 * 2 * (size_t)(nr + 2) * t.NGB);
    t.o_row = take(4 * (size_t)(2 * nr + 4));
    t.o_need = take(4 * 6 * (size_t)nr);
    t.bytes = o;
    return t;
}

template <int RHO>
// filter: apply Eq. 15-16 (0: the image is used as it is, the median pre-filter's output or bilateral = 0)
__device__ __forceinline__ void grad_body(const KParams &kp, const Work &w, const float *__restrict__ disp,
                                          const uint8_t *__restrict__ img, int R, const int f, const int bx, const int by,
                                          const bool filter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NW = kWarps;
    const int W = kp.W, H = kp.H, NG = (W + 3) >> 2;
    const int r0 = by * R, nr = min(R, H - r0);
    const int j0 = bx * kGroups, nj = min(kGroups, NG - j0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const FrameState &fs = w.fs[f];
    const int vtop = fs.v_top;
    if ((fs.flags & LD_F_NO_LANES) || r0 + nr - 1 < vtop)
        return;   // no road pixel of the tile (k_vdisp zeroed the per-row counts)
    if (!LD_IN(kp.n_cls, kClsTables + 1, CK_GRAD_TILE))   // the class tables the tile copies
        return;
    const GradTile T = grad_tile<RHO>(nr, nj, kp.n_cls);
    const int cbase = 4 * j0 - RHO - 4, rbase = r0 - RHO - 1;   // frame column / row of tile column / row 0
    uint16_t *tabs = reinterpret_cast<uint16_t *>(smem + T.o_tab);    // [n_cls][512]
    uint16_t *tile = reinterpret_cast<uint16_t *>(smem + T.o_tile);   // [TR][TWP] 2 I, or 2 x sentinel
    uint32_t *rng = reinterpret_cast<uint32_t *>(smem + T.o_ibf);     // [nr][NB] (min 2 I, 1022 - max 2 I) of a block's windows
    uint8_t *live = smem + T.o_live;                                  // [nr][IWO] owned road pixels left after pruning
    uint8_t *ibf = smem + T.o_ibf;                                    // [nr + 2][IWB] bilateral output, row b = v - r0 + 1
    // pixel pairs (b << 8 | half << 7 | g) that need the filter, and [nr][2][3] the left and right pairs of the
    // bilateral groups that a row's Sobel reads
    uint16_t *glist = reinterpret_cast<uint16_t *>(smem + T.o_gl);
    uint32_t *needm = reinterpret_cast<uint32_t *>(smem + T.o_need);
    float *rowVy = reinterpret_cast<float *>(smem + T.o_row);
    int *cnt = reinterpret_cast<int *>(rowVy + 2 * nr);               // [1] pairs that need the filter

    // per-class weight tables T_c[a] = (ws_c * wr(a) + 2^14) >> 15 for a = |I(i,j) - I(u,v)|, built once per
    // handle (zero from a = 256 on), copied asynchronously in 16-byte pieces (cp.async): the filter is the
    // first reader, so the copy overlaps the staging, flatness and compaction phases
    {
        const int nt16 = kp.n_cls * (kTabBytes / 16);
        const char *src = reinterpret_cast<const char *>(w.cls_tab);
        const uint32_t dst0 = smem_addr(tabs);
        for (int k = tid; k < nt16; k += kThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst0 + 16u * (uint32_t)k),
                         "l"(src + 16 * (size_t)k) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const float *rows = w.rows + (size_t)f * 3 * H;
    if (tid < nr)
        rowVy[tid] = __ldg(rows + H + r0 + tid);   // V_py(v) of the owned rows, for the votes
    if (tid == 0)
        *cnt = 0;
    // road mask of the owned pixels first: l > 0 with |l - f(v)| <= varpi (an infinite or NaN l fails the
    // second test because f(v) is finite), v >= v_top, 1 <= u <= W-2.  A warp takes two rows at a time with
    // all of their loads in flight, f(v) read directly (rows off the road get NaN, which fails the test).
    const float *dsrc = disp + ((size_t)f * H + r0) * W;
    constexpr int KX = 4 * kGroups / 32;   // 32-pixel chunks of an owned row
    for (int rr = 2 * warp; rr < nr; rr += 2 * NW) {
        float lv[2][KX], fv[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int r = rr + q, v = r0 + r;
            fv[q] = r < nr && v >= vtop && v >= 1 && v <= H - 2 ? __ldg(rows + v) : __int_as_float(0x7fc00000);
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                const int u = 4 * j0 + lane + 32 * k;
                lv[q][k] = r < nr && lane + 32 * k < T.IWO && u >= 1 && u <= W - 2 ? __ldg(dsrc + (size_t)r * W + u)
                                                                                    : 0.0f;
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                const int r = rr + q, x = lane + 32 * k;
                if (r < nr && x < T.IWO)
                    live[r * T.IWO + x] = (uint8_t)(lv[q][k] > 0.0f && fabsf(__fsub_rn(lv[q][k], fv[q])) <= kp.varpi);
            }
    }
    // image region, four pixels a lane: a row starts at any byte, so a lane takes the two aligned words its pixels
    // lie in and shifts.  (Words that are not wholly inside the frame's bytes are put together from byte loads; the
    // pixels beside the frame's columns, which such a word also reads, become the sentinel.)  A warp takes two tile
    // rows at a time and issues all of their loads before its first store.
    const uint8_t *im = img + (size_t)f * H * W;
    const uintptr_t fb = reinterpret_cast<uintptr_t>(im), fe = fb + (size_t)H * W;
    const bool edge_tile = cbase < 0 || cbase + T.TWP > W;
    constexpr int KC = (4 * kGroups + 2 * RHO + 11 + 127) / 128;   // 32-word chunks of a tile row
    for (int tr0 = 2 * warp; tr0 < T.TR; tr0 += 2 * NW) {
        uint32_t px[2][KC];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int v = rbase + tr0 + q;
            const bool vin = tr0 + q < T.TR && v >= 0 && v < H;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int tc = 4 * (lane + 32 * k);
                px[q][k] = 0u;
                if (vin && tc < T.TWP) {
                    const uintptr_t a = fb + (ptrdiff_t)v * W + cbase + tc, a4 = a & ~(uintptr_t)3;
                    if (a4 >= fb && a4 + 8 <= fe) {
                        const uint32_t *src = reinterpret_cast<const uint32_t *>(a4);
                        px[q][k] = __funnelshift_r(__ldg(src), __ldg(src + 1), 8u * (uint32_t)(a & 3));
                    } else {
                        for (int p = 0; p < 4; ++p)
                            if (a + p >= fb && a + p < fe)
                                px[q][k] |= (uint32_t)__ldg(reinterpret_cast<const uint8_t *>(a + p)) << (8 * p);
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int v = rbase + tr0 + q;
            const bool vin = v >= 0 && v < H;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int tc = 4 * (lane + 32 * k), c = cbase + tc;
                uint32_t lo = 2u * __byte_perm(px[q][k], 0u, 0x4140), hi = 2u * __byte_perm(px[q][k], 0u, 0x4342);
                if (edge_tile || !vin) {
                    const uint32_t out = 2u * kSentinel;
                    lo = vin && (unsigned)c < (unsigned)W ? lo : (lo & 0xffff0000u) | out;
                    lo = vin && (unsigned)(c + 1) < (unsigned)W ? lo : (lo & 0xffffu) | out << 16;
                    hi = vin && (unsigned)(c + 2) < (unsigned)W ? hi : (hi & 0xffff0000u) | out;
                    hi = vin && (unsigned)(c + 3) < (unsigned)W ? hi : (hi & 0xffffu) | out << 16;
                }
                if (tr0 + q < T.TR && tc < T.TWP)
                    *reinterpret_cast<uint2 *>(tile + (tr0 + q) * T.TWP + tc) = make_uint2(lo, hi);
            }
        }
    }
    __syncthreads();
    // Exact pruning (see the comment at the top): a group is flat when the image range over its test window, a
    // superset of its 3x3 neighbours' windows (kFlatBlocks four-column blocks from tile column 4 (g - j0), rows
    // v - RHO - 1 .. v + RHO + 1), is at most kp.flat_range; any tap outside the frame holds the sentinel, which
    // makes the range too large.  A pair (min 2 I, 1022 - max 2 I) is one 32-bit word whose halves are both minimised
    // by one instruction.  Here a thread takes one block column and kFlatRows rows: the pairs of its rows, then
    // window minima over doubling numbers of rows.
    if (kp.flat_range >= 0) {
        constexpr int WN = 2 * RHO + 3, NI = kFlatRows + WN - 1;       // window rows, rows read
        constexpr int K = WN >= 8 ? 8 : 4;                              // the largest power of two up to WN
        const int tasks = T.NB * ((nr + kFlatRows - 1) / kFlatRows);
        for (int t = tid; t < tasks; t += kThreads) {
            const int seg = t / T.NB, blk = t - seg * T.NB, ra = seg * kFlatRows;
            const uint16_t *src = tile + ra * T.TWP + 4 * blk;
            uint32_t m[NI];
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const uint2 v = ra + i < T.TR ? *reinterpret_cast<const uint2 *>(src + i * T.TWP) : make_uint2(0u, 0u);
                const uint32_t mn = __vminu2(v.x, v.y), mx = __vmaxu2(v.x, v.y);
                m[i] = __vminu2(__byte_perm(mn, 0x03fe03feu - mx, 0x5410), __byte_perm(mn, 0x03fe03feu - mx, 0x7632));
            }
#pragma unroll
            for (int d = 1; d < K; d *= 2)
#pragma unroll
                for (int i = 0; i + d < NI; ++i)
                    m[i] = __vminu2(m[i], m[i + d]);
#pragma unroll
            for (int i = 0; i < kFlatRows; ++i)
                if (ra + i < nr)
                    rng[(ra + i) * T.NB + blk] = __vminu2(m[i], m[i + WN - K]);
        }
        __syncthreads();
    }
    // flat groups leave the mask; then, per row, the pixel pairs of the bilateral groups g' = j0 - 1 + g (g < NGB,
    // 66 bits each for the left and the right pairs) that the Sobel of a remaining road pixel reads
    for (int r = warp; r < nr; r += NW) {
        uint64_t lp = 0, rp = 0, first = 0, last = 0;   // groups whose left / right pair, previous or next pair is read
#pragma unroll
        for (int h = 0; h < kGroups / 32; ++h) {
            const int g = lane + 32 * h;
            uint32_t lw = 0u;
            if (g < nj) {
                lw = reinterpret_cast<const uint32_t *>(live + r * T.IWO)[g];
                if (kp.flat_range >= 0) {
                    const uint32_t *src = rng + r * T.NB + g;
                    uint32_t m = src[0];
#pragma unroll
                    for (int k = 1; k < kFlatBlocks<RHO>; ++k)
                        m = __vminu2(m, src[k]);
                    if (1022 - (int)((m >> 16) + (m & 0xffffu)) <= 2 * kp.flat_range) {
                        lw = 0u;
                        reinterpret_cast<uint32_t *>(live + r * T.IWO)[g] = 0u;
                    }
                }
            }
            lp |= (uint64_t)__ballot_sync(0xffffffffu, (lw & 0xffffffu) != 0u) << (32 * h);
            rp |= (uint64_t)__ballot_sync(0xffffffffu, (lw >> 8) != 0u) << (32 * h);
            first |= (uint64_t)__ballot_sync(0xffffffffu, (lw & 0xffu) != 0u) << (32 * h);
            last |= (uint64_t)__ballot_sync(0xffffffffu, (lw >> 24) != 0u) << (32 * h);
        }
        if (lane < 6) {
            const bool right = lane >= 3;
            const int k = right ? lane - 3 : lane;
            const uint64_t lo = right ? (rp << 1) | first : (lp << 1) | (last << 2);
            const uint64_t hi = right ? rp >> 63 : (lp >> 63) | (last >> 62);
            needm[6 * r + lane] = k == 2 ? (uint32_t)hi : (uint32_t)(lo >> (32 * k));
        }
    }
    __syncthreads();
    // the pairs of rows v = r0 - 1 + b (b < nr + 2): those of road rows b - 2 .. b, 32 groups a thread
    for (int t0 = 0; t0 < 3 * (nr + 2); t0 += kThreads) {
        const int t = t0 + tid, b = t / 3, k = t - 3 * b;
        uint32_t ml = 0u, mr = 0u;
        if (t < 3 * (nr + 2)) {
#pragma unroll
            for (int dr = 0; dr < 3; ++dr)
                if (b - dr >= 0 && b - dr < nr) {
                    ml |= needm[6 * (b - dr) + k];
                    mr |= needm[6 * (b - dr) + 3 + k];
                }
        }
        const int n = __popc(ml) + __popc(mr);
        int at = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, at, d);
            at += lane >= d ? o : 0;
        }
        int base = 0;
        if (lane == 31 && at)
            base = atomicAdd(cnt, at);
        at += __shfl_sync(0xffffffffu, base, 31) - n;
        for (uint32_t m = ml | mr; m; m &= m - 1) {
            const int bit = __ffs(m) - 1, e = (b << 8) | (32 * k + bit);
            if ((ml >> bit) & 1u) {
                if (LD_IN(at, 2 * (nr + 2) * T.NGB, CK_GRAD_GLIST))
                    glist[at] = (uint16_t)e;
                ++at;
            }
            if ((mr >> bit) & 1u) {
                if (LD_IN(at, 2 * (nr + 2) * T.NGB, CK_GRAD_GLIST))
                    glist[at] = (uint16_t)(e | 128);
                ++at;
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");   // this thread's table pieces have landed
    __syncthreads();
    const int ng = LD_IN(*cnt, 2 * (nr + 2) * T.NGB + 1, CK_GRAD_GLIST) ? *cnt : 0;
    const uint32_t tab = smem_addr(tabs);
    for (int k = tid; k < ng; k += kThreads) {
        const int e = glist[k], b = e >> 8, g = e & 127, c = 4 * g + ((e >> 6) & 2);
        // the pair's cell, then its windows (tile rows b .. b + 2 RHO, tile columns c .. c + 2 RHO + 1)
        if (!LD_IN(b, nr + 2, CK_GRAD_GROUP) || !LD_IN(g, T.NGB, CK_GRAD_GROUP) ||
            !LD_IN(b + 2 * RHO, T.TR, CK_GRAD_TAP) || !LD_IN(c + 2 * RHO + 1, T.TWP, CK_GRAD_TAP))
            continue;
        const int u0 = 4 * (j0 - 1) + c, v = r0 - 1 + b;   // frame column of the pair, frame row
        const int nv = min(2, W - u0);
        uint32_t out;
        // the pair's windows start at tile row b (frame row v - RHO) and tile column c (frame column u0 - RHO)
        if (filter) {
            out = bilateral2<RHO>(tile, T.TWP, b, c, nv, tab);
        } else {
            const uint16_t *src = tile + (b + RHO) * T.TWP + c + RHO;
            out = (uint32_t)(src[0] >> 1) | ((uint32_t)(src[1] >> 1) << 8);
        }
        *reinterpret_cast<uint16_t *>(ibf + b * T.IWB + c) = (uint16_t)out;
        if (w.dbg_ibf && v >= 0 && v < H && u0 >= 0) {   // stage capture (pairs shared with other tiles too)
            int16_t *drow = w.dbg_ibf + ((size_t)f * H + v) * W;
            for (int q = 0; q < nv; ++q)
                drow[u0 + q] = (int16_t)((out >> (8 * q)) & 0xffu);
        }
    }
    __syncthreads();

    // Sobel, edge test, votes of the remaining owned road pixels, a warp per row.  A lane takes a group's four
    // pixels from 32-bit loads of the mask and of the three bilateral rows (owned group g is bilateral group
    // g + 1), two pixels per 32-bit operation; the edge pixels go to the warp's list in shared memory, so the
    // division, the appends (one atomic per row and list) and their stores run on full warps.
    const int thr2 = kp.edge_thresh2;
    int16_t *edges = w.edges + (size_t)f * H * W * 4;
    int16_t *vbins = w.vbins + (size_t)f * H * W;
    int32_t *ecnt = w.ecount + (size_t)f * H;
    int32_t *vcnt = w.vcount + (size_t)f * H;
    short4 *list = reinterpret_cast<short4 *>(smem + T.o_tile) + warp * T.IWO;   // (u, -, G_x, G_y); warps >= nr: unused
    int16_t *blist = reinterpret_cast<int16_t *>(list);                          // vote columns, over entries already read
    const unsigned below = (1u << lane) - 1u;
    for (int r = warp; r < nr; r += NW) {
        const int v = r0 + r;
        int tot = 0;
#pragma unroll
        for (int g0 = 0; g0 < kGroups; g0 += 32) {
            const int g = g0 + lane;
            const uint32_t m4 = g < nj ? reinterpret_cast<const uint32_t *>(live + r * T.IWO)[g] : 0u;
            if (!__any_sync(0xffffffffu, m4 != 0u))
                continue;
            int gx[4] = {}, gy[4] = {};
            if (m4) {
                // columns -1 .. 4 of the group as 16-bit pairs: e = (-1, 1), o = (0, 2), f = (1, 3), q = (2, 4)
                uint32_t e[3], o[3], ff[3], q[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const uint32_t *rw = reinterpret_cast<const uint32_t *>(ibf + (r + d) * T.IWB) + g;
                    const uint32_t x0 = rw[0], x1 = rw[1], x2 = rw[2];
                    const uint32_t a4 = __funnelshift_r(x0, x1, 24), b4 = __funnelshift_r(x1, x2, 8);
                    e[d] = a4 & 0x00ff00ffu;
                    o[d] = (a4 >> 8) & 0x00ff00ffu;
                    ff[d] = b4 & 0x00ff00ffu;
                    q[d] = (b4 >> 8) & 0x00ff00ffu;
                }
                // G_x: column sums (1, 2, 1) right minus left; G_y: row sums (1, 2, 1) below minus above; every half
                // is 1024 + value, in [4, 2044], so no half borrows from the other
                const uint32_t bias = 0x04000400u;
                const uint32_t gx02 = (ff[0] + 2u * ff[1] + ff[2]) + bias - (e[0] + 2u * e[1] + e[2]);
                const uint32_t gx13 = (q[0] + 2u * q[1] + q[2]) + bias - (o[0] + 2u * o[1] + o[2]);
                const uint32_t gy02 = (e[2] + 2u * o[2] + ff[2]) + bias - (e[0] + 2u * o[0] + ff[0]);
                const uint32_t gy13 = (o[2] + 2u * ff[2] + q[2]) + bias - (o[0] + 2u * ff[0] + q[0]);
                gx[0] = (int)(gx02 & 0xffffu) - 1024;
                gx[1] = (int)(gx13 & 0xffffu) - 1024;
                gx[2] = (int)(gx02 >> 16) - 1024;
                gx[3] = (int)(gx13 >> 16) - 1024;
                gy[0] = (int)(gy02 & 0xffffu) - 1024;
                gy[1] = (int)(gy13 & 0xffffu) - 1024;
                gy[2] = (int)(gy02 >> 16) - 1024;
                gy[3] = (int)(gy13 >> 16) - 1024;
            }
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const bool edge = ((m4 >> (8 * p)) & 0xffu) != 0u && gx[p] * gx[p] + gy[p] * gy[p] > thr2;
                const unsigned m = __ballot_sync(0xffffffffu, edge);
                if (edge)
                    list[tot + __popc(m & below)] = make_short4((short)(4 * (j0 + g) + p), 0, (short)gx[p], (short)gy[p]);
                tot += __popc(m);
            }
        }
        if (!tot)
            continue;
        int pe = 0;
        if (lane == 0)
            pe = atomicAdd(ecnt + v, tot);
        __syncwarp();
        const float av = __fsub_rn((float)v, rowVy[r]);
        pe = __shfl_sync(0xffffffffu, pe, 0);
        short4 *dst = reinterpret_cast<short4 *>(edges) + (size_t)v * W + pe;
        int nb = 0;
        for (int k0 = 0; k0 < tot; k0 += 32) {
            const int k = k0 + lane;
            int bin = -1;
            if (k < tot) {
                short4 en = list[k];
                if (en.z != 0) {
                    const float bv = __fmul_rn(av, (float)en.w);
                    const float qv = __fdiv_rn(bv, (float)en.z);
                    const float vs = __fadd_rn((float)en.x, qv);
                    const float col = floorf(__fadd_rn(vs, 0.5f));
                    if (col >= 0.0f && col < (float)W)
                        bin = (int)col;
                }
                en.y = (short)bin;
                if (LD_IN(pe + k, W, CK_GRAD_EDGE))   // a row holds at most W edge entries
                    dst[k] = en;
            }
            const unsigned m = __ballot_sync(0xffffffffu, bin >= 0);   // (and the list's reads are done)
            if (bin >= 0)
                blist[nb + __popc(m & below)] = (int16_t)bin;
            nb += __popc(m);
        }
        if (nb) {
            int pv = 0;
            if (lane == 0)
                pv = atomicAdd(vcnt + v, nb);
            pv = __shfl_sync(0xffffffffu, pv, 0);
            __syncwarp();
            for (int k = lane; k < nb; k += 32) {
                const int bin = blist[k];
                if (LD_IN(pv + k, W, CK_GRAD_VOTE) && LD_IN(bin, W, CK_GRAD_VOTE))
                    vbins[(size_t)v * W + pv + k] = (int16_t)bin;
            }
        }
        __syncwarp();   // the list is free for the warp's next row
    }
}

template <int RHO>
__global__ void __launch_bounds__(kThreads, 4) k_grad(const KParams kp, const Work w, const float *__restrict__ disp,
                                                   const uint8_t *__restrict__ img, int R)
{
    grad_body<RHO>(kp, w, disp, img, R, blockIdx.y, blockIdx.x, gridDim.z - 1 - blockIdx.z, kp.bilateral != 0);
}

// median_input: the frame's image is its median-filtered copy in the workspace (bilateral = 2)
template <int RHO>
__global__ void __launch_bounds__(kThreads, 4) k_grad_fd(const FrameDesc *__restrict__ fd, int R, int median_input)
{
    const FrameDesc &d = fd[blockIdx.y];
    const KParams kp = d.kp;   // the frame's parameters, loaded once into registers
    const Work w = d.w;
    const int by = gridDim.z - 1 - blockIdx.z;
    if (by * R >= kp.H || (int)blockIdx.x * kGroups >= (kp.W + 3) / 4)
        return;
    grad_body<RHO>(kp, w, d.disp, median_input ? w.med : d.img, R, 0, blockIdx.x, by,
                   !median_input && kp.bilateral != 0);
}

// Rows per CTA: the tuned value when set, else 16.
template <int RHO>
int grad_rows(int tuned)
{
    return tuned > 0 ? (tuned < 64 ? tuned : 64) : 16;
}

template <int RHO>
cudaError_t launch_grad_t(const KParams &kp, const Work &w, const float *disp, const uint8_t *img, cudaStream_t s)
{
    const int R = grad_rows<RHO>(kp.tile_grad);
    const int NG = (kp.W + 3) / 4, nj = NG < kGroups ? NG : kGroups;
    const size_t smem = grad_tile<RHO>(R, nj, kp.n_cls).bytes;
    dim3 grid((NG + kGroups - 1) / kGroups, kp.n_frames, (kp.H + R - 1) / R);
    k_grad<RHO><<<grid, kThreads, smem, s>>>(kp, w, disp, img, R);
    return cudaGetLastError();
}

template <int RHO>
cudaError_t launch_grad_fd_t(const KParams &kmax, const FrameDesc *fd, int n, bool median_input, cudaStream_t s)
{
    const int R = grad_rows<RHO>(0);
    const int NG = (kmax.W + 3) / 4, nj = NG < kGroups ? NG : kGroups;
    const size_t smem = grad_tile<RHO>(R, nj, kmax.n_cls).bytes;
    dim3 grid((NG + kGroups - 1) / kGroups, n, (kmax.H + R - 1) / R);
    k_grad_fd<RHO><<<grid, kThreads, smem, s>>>(fd, R, median_input ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_grad_fd(const KParams &kmax, const FrameDesc *fd, int n, bool median_input, cudaStream_t s)
{
    switch (kmax.rho) {
    case 1: return launch_grad_fd_t<1>(kmax, fd, n, median_input, s);
    case 2: return launch_grad_fd_t<2>(kmax, fd, n, median_input, s);
    case 3: return launch_grad_fd_t<3>(kmax, fd, n, median_input, s);
    case 4: return launch_grad_fd_t<4>(kmax, fd, n, median_input, s);
    default: return launch_grad_fd_t<5>(kmax, fd, n, median_input, s);
    }
}

cudaError_t setup_grad(int smem_optin)
{
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad<1>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad<2>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad<3>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad<4>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad<5>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad_fd<1>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad_fd<2>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad_fd<3>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad_fd<4>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_grad_fd<5>, smem_optin);
    return e;
}

cudaError_t launch_grad(const KParams &kp, const Work &w, const float *disp, const uint8_t *img, cudaStream_t s)
{
    switch (kp.rho) {
    case 1: return launch_grad_t<1>(kp, w, disp, img, s);
    case 2: return launch_grad_t<2>(kp, w, disp, img, s);
    case 3: return launch_grad_t<3>(kp, w, disp, img, s);
    case 4: return launch_grad_t<4>(kp, w, disp, img, s);
    default: return launch_grad_t<5>(kp, w, disp, img, s);
    }
}

}  // namespace ld
