// k_vpx_dp, one CTA per frame (Sec. 2.3.2-2.3.3): the dense accumulator m_x (Alg. 5) as a sliding band of
// vote rows, and Eq. 18 from row H-1 up to v_top,
//   E_v(u) = m_x(u, v) + min_{tau in [-tau_x, tau_x], 0 <= u + tau < W} [E_{v+1}(u + tau) + lambda_x |tau|],
// the path M_x = {(v, u_v)} by backtracking, and the path points whose cell holds votes, for the RANSAC fit.
//
// Readings: Eq. 18's "+lambda_x tau" is read as lambda_x |tau|.  Ties take the smaller |tau|, then the
// negative one; the path starts at the smallest index minimising its last row.  Alg. 5 is read from the text
// around it: m_x(u, j) = -varrho * (votes in column u of rows [j - chi, j + chi] within [v_top, H-1]).  A
// path point whose cell holds no count carries no observation.
//
// The rows follow one another, so the time is rows x (time of a row), and a row is bound by integer
// instructions (two cycles each per scheduler) and by its chain of latencies.  Layout:
//   - four DP warps (eight past 2400 columns, 2560 with tau_x = 0), one per scheduler, hold the row in registers, kCells adjacent
//     cells per lane.  A warp's range overlaps its neighbours' by `halo` lanes on each side: a row spoils
//     tau_x cells at either end, so `rows` rows pass before the warps exchange their edge cells through
//     shared memory and meet at a barrier (instead of one barrier and a shared-memory window per row);
//   - candidates are keys 16 (E + lambda_x |tau|) + rank in tie order (0, -1, +1, -2, ...), so the tie-broken
//     argmin is an integer minimum.  The keys' penalty is linear in |tau| on either side (c = 16 lambda_x + 2
//     a step, the left side one less), so minima over three adjacent steps, g, serve all cells: two
//     three-way minima and two to three more per cell instead of 2 tau_x.  The g that a neighbouring lane
//     needs come from this lane's own cells, so one round of shuffles serves a row; it is issued at the end
//     of the row before, ahead of packing and storing that row's ranks;
//   - four producer warps scatter the band changes (votes of the row entering and of the row leaving the
//     band, read from the gradient kernel's lists) of the next `rows` rows into a ring of shared-memory rows
//     while the DP warps work;
//   - columns off the frame are cells that pay an extra penalty per row: a path through one costs more than
//     the path that stays in the frame's edge column, so they never win and need no test.
// The ranks go to global memory (L2-resident; the frame's part of M_1, not yet written), a byte per cell with a bit that says whether the
// cell holds votes; a row is stored in planes of one word (four cells) per lane, so that every store of a warp
// is contiguous.  The backtrack walks blocks of 32 rows: the other warps fetch the columns that the next block
// can reach and turn their ranks into displacements, so that a step of the walk is one shared-memory load and
// one addition.
//
// Measured (GB300), against two cells per thread with a barrier and a shared-memory window of the row per DP row:
// 64 x 1242x375 154 -> 100 us, one such frame 149 -> 92, 16 x 1920x1080 573 -> 330, one 320x120 frame 39 -> 31.  A
// row of 1242 columns takes about 570 cycles (12 cells a lane, an exchange every 7 rows), of which the
// instructions of 12 cells are about 390; the backtrack is about 100 cycles a row.
#include <type_traits>

#include "k_dp.cuh"

namespace ld {

namespace {

constexpr int kProducers = 4;
constexpr int kMaxCells = 20;               // cells per lane at most
constexpr int kMaxRows = 8;                 // rows between two exchanges at most
constexpr size_t kRingBytes = 160 * 1024;   // band changes of 2 * rows rows
constexpr int kBlock = 32;                  // rows of a backtrack block
constexpr uint32_t kHasVotes = 0x80;        // bit of a cell's byte in a backtrack row, beside the rank: the band key's sign
constexpr int kOffKey = 1 << 29;            // key of a column off the frame on the first row (others are at most 0)
constexpr int kOffRow = 16 * 64;            // and what it pays per row
// Keys fit 32 bits while 16 |E| does.  The number of a frame's votes settles it for almost every frame (each vote is in at
// most 2 chi + 1 bands), but most of the frames beyond that fit too, since their votes do not lie in one column.  So in
// those every exchange looks at the keys: above kKeyFloor, the rows up to the next one cannot leave the range.  Once a key
// is below, keys are held at the floor and the result is dropped.  A row lowers a key by at most 16 varrho m, and a cell's
// m is at most W times the smaller of H and 2 chi + 1.  ld_create requires varrho (2 chi + 1) W H < 2^30: with
// H >= 16 kMaxRows, kMaxRows rows lower a key by less than 2^30, and with a smaller H by at most 16 kMaxRows 16 W H, less
// than 2^30 as well.  Texture all over 64 frames of 1242 x 375, varrho 16, chi 64: the call takes 864 us; 1579 when every
// frame whose votes could pass 2^25 went to vpx_forward_wide.
constexpr int kKeyFloor = -((1 << 30) - (1 << 20));
static_assert(16LL * kMaxRows * kMaxVoteRho * LD_MAX_W * (16 * kMaxRows - 1) <= 1LL << 30, "rows between two looks at the keys");

__device__ __forceinline__ int lds_s8(uint32_t a)
{
    int v;
    asm volatile("ld.shared.s8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
// Vector accesses by shared address: the carved pointers are generic to the compiler, whose accesses take
// longer than the shared ones.
__device__ __forceinline__ int4 lds4(uint32_t a)
{
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts4(uint32_t a, int4 v)
{
    asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts1(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// What the kernel reads of a frame's parameters and workspace.
struct VpxArgs {
    int W, H, chi, vote_rho, lambda_x, tau_x, band_literal;
    int pmax;
    const FrameState *fs;
    const int32_t *vcount;
    const int16_t *vbins;
    int32_t *M1;          // holds the backtrack rows here
    int16_t *path_x, *pts;
    int32_t *npts, *dbg_mx;
};
__host__ __device__ inline VpxArgs vpx_args(const KParams &kp, const Work &w)
{
    return {kp.W, kp.H, kp.chi, kp.vote_rho, kp.lambda_x, kp.tau_x, kp.band_literal, w.pmax,
            w.fs, w.vcount, w.vbins, w.M1, w.path_x, w.pts, w.npts, w.dbg_mx};
}

// How a row of W cells lies on the DP warps (vpx_plan).
struct VpxPlan {
    int cells;    // per lane
    int warps;    // DP warps
    int halo;     // lanes shared with each neighbour
    int rows;     // rows between exchanges: tau_x * rows <= halo * cells
    int own;      // cells a warp owns: (32 - 2 halo) * cells
    int stride;   // ints of a ring row: every warp's cells, from column -halo * cells
};

// Shared-memory layout of k_vpx_dp.
struct VpxMem {
    int16_t *cnt;          // [H] votes per row (0 above v_top)
    int16_t *path;         // [H]
    uint8_t *sup;          // [H]
    int *sh;
    int16_t *pid;          // [H]
    int *box;              // [2][warps][2][halo * cells] edge cells: for the left and for the right neighbour
    // one space, used in turn: [2 rows + 1][stride] band changes (column u at halo * cells + u; the last row
    // is only loaded ahead), then the backtrack windows
    int *ring;
};

__device__ __forceinline__ const int16_t *vote_list(const VpxArgs &a, int f, int r)
{
    return a.vbins + ((size_t)f * a.H + r) * a.W;
}
// Adds `by` for every vote of row r from its q0-th on to the counts at shared address `to`, by the threads t0,
// t0 + stride, ...; a row holds anything from none to a thousand votes, eight loads in flight.
__device__ __forceinline__ void add_votes(const VpxArgs &a, const VpxMem &S, int f, int r, int q0, uint32_t to, int by, int t0,
                                          int stride)
{
    const int n = S.cnt[r];
    const int16_t *list = vote_list(a, f, r);
    for (int q = q0 + t0; q < n; q += 8 * stride) {
        int c[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            c[k] = q + k * stride < n ? (int)__ldg(list + q + k * stride) : -1;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (c[k] >= 0 && LD_IN(c[k], a.W, CK_VPX_VOTE))
                atoms_add(to + 4u * (uint32_t)c[k], by);
    }
}

// Scatter the band change between row v+1 and row v (votes of row v - chi enter, of row v + chi + 1 leave)
// into the delta array `delta` (shared address of column 0) as +unit and -unit, by the threads t0, t0 + stride, ...
__device__ __forceinline__ void scatter_delta(const VpxArgs &a, const VpxMem &S, int f, int v, int vtop, uint32_t delta, int unit,
                                              int t0, int stride)
{
    const int vmax = a.H - 1, chi = a.chi;
    if (a.band_literal && v >= vmax - chi - 1) {
        // band_literal_bottom: rows j > vmax - chi - 1 use the band [j, vmax], so there row v enters and
        // nothing leaves; at v = vmax - chi - 1 the band [v - chi, v + chi] replaces [v + 1, vmax]
        const int r_lo = v >= vmax - chi ? v : max(vtop, v - chi);
        for (int r = max(r_lo, vtop); r <= v; ++r)
            add_votes(a, S, f, r, 0, delta, unit, t0, stride);
        if (v == vmax - chi - 1)
            add_votes(a, S, f, vmax, 0, delta, -unit, t0, stride);
        return;
    }
    if (v - chi >= vtop)
        add_votes(a, S, f, v - chi, 0, delta, unit, t0, stride);
    if (v + chi + 1 <= vmax)
        add_votes(a, S, f, v + chi + 1, 0, delta, -unit, t0, stride);
}

// Byte of cell u in a backtrack row of cells-wide lanes: plane (u % cells) / 4 of one word per lane.  The rows lie in the
// frame's part of M_1, from its first 16-byte boundary on (k_m1 writes it two stages later).  H rows fit its 4 W H bytes
// at every width and its layout (16 columns: 32 bytes a row); a narrow frame that shares a launch, and so the layout, with
// wide ones has a slot of the widest one's size.
__host__ __device__ constexpr int bt_plane(int W, int cells) { return 4 * (((W + cells - 1) / cells + 3) & ~3); }
__host__ __device__ constexpr int bt_row(int W, int cells) { return bt_plane(W, cells) * (cells / 4); }
__device__ __forceinline__ int bt_byte(int u, int cells, int plane)
{
    const int g = u / cells, x = u - g * cells;
    return (x >> 2) * plane + 4 * g + (x & 3);
}

// A warp's cells of one row: the keys f, and what the next row needs of the neighbouring lanes.
template <int TAU, int C>
struct DpRow {
    static constexpr int K = TAU > 2 ? TAU - 2 : 0;   // farthest start of a three-step window
    static_assert(C >= K + 2, "a lane's shuffled windows come from its own cells");
    int f[C];
    int before[2], after[2];                          // keys of cells -2, -1 and C, C + 1
    int gl[C + K], gr[C + K];                         // gl[x + K]: cell x = -K .. C - 1; gr[x]: cell x = 0 .. C + K - 1

    __device__ __forceinline__ int key(int x) const { return x < 0 ? before[x + 2] : x < C ? f[x] : after[x - C]; }
    // minima over steps 0 .. 2 to the left and to the right of cell x
    __device__ __forceinline__ int left(int x, int c) const { return __vimin3_s32(key(x), key(x - 1) + c, key(x - 2) + 2 * c); }
    __device__ __forceinline__ int right(int x, int c) const { return __vimin3_s32(key(x), key(x + 1) + c, key(x + 2) + 2 * c); }

    // exchange with the neighbouring lanes
    __device__ __forceinline__ void edges(int c)
    {
        constexpr unsigned kAll = 0xffffffffu;
        if constexpr (TAU > 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                gl[C + k] = left(C - K + k, c);
                gr[k] = right(k, c);
            }
            before[1] = __shfl_up_sync(kAll, f[C - 1], 1);
            after[0] = __shfl_down_sync(kAll, f[0], 1);
            if constexpr (TAU > 1) {
                before[0] = __shfl_up_sync(kAll, f[C - 2], 1);
                after[1] = __shfl_down_sync(kAll, f[1], 1);
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                gl[k] = __shfl_up_sync(kAll, gl[C + k], 1);
                gr[C + k] = __shfl_down_sync(kAll, gr[k], 1);
            }
        }
    }
    // the candidates' minima of the next row (16 (E + penalty) + rank)
    __device__ __forceinline__ void minima(int c, int *best)
    {
        if constexpr (TAU == 0) {
#pragma unroll
            for (int x = 0; x < C; ++x)
                best[x] = f[x];
        } else if constexpr (TAU == 1) {
#pragma unroll
            for (int x = 0; x < C; ++x)
                best[x] = __viaddmin_s32(key(x - 1), c - 1, __viaddmin_s32(key(x + 1), c, f[x]));
        } else if constexpr (TAU == 2) {
#pragma unroll
            for (int x = 0; x < C; ++x)
                best[x] = __viaddmin_s32(key(x - 2), 2 * c - 1, __viaddmin_s32(key(x - 1), c - 1,
                          __viaddmin_s32(key(x + 2), 2 * c, __viaddmin_s32(key(x + 1), c, f[x]))));
        } else {
#pragma unroll
            for (int x = 0; x < C - K; ++x)
                gl[x + K] = left(x, c);
#pragma unroll
            for (int x = K; x < C; ++x)
                gr[x] = right(x, c);
            // windows of steps s .. s + 2: to the right from 0, to the left from 1, the last ending at TAU
            constexpr int nL = (TAU + 2) / 3, nR = (TAU + 3) / 3;
#pragma unroll
            for (int x = 0; x < C; ++x) {
                int b = gr[x];
#pragma unroll
                for (int i = 1; i < nR; ++i) {
                    const int s = 3 * i < K ? 3 * i : K;
                    b = __viaddmin_s32(gr[x + s], s * c, b);
                }
#pragma unroll
                for (int i = 0; i < nL; ++i) {
                    const int s = 1 + 3 * i < K ? 1 + 3 * i : K;
                    b = __viaddmin_s32(gl[x + K - s], s * c - 1, b);
                }
                best[x] = b;
            }
        }
    }
};

// The forward DP with packed keys.  Returns the first column minimising row vtop to every thread, or -1 when the keys
// passed kKeyFloor (looked for when LOOK).
template <int TAU, int C, bool LOOK>
__device__ __forceinline__ int vpx_forward(const VpxArgs &a, const VpxMem &S, const VpxPlan &P, int f, int vtop, uint8_t *gbt)
{
    const int W = a.W, vmax = a.H - 1, RB = bt_row(W, C);
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int R = P.rows, HL = P.halo, HC = HL * C, stride = P.stride;
    const bool dp = warp < P.warps;
    const int scale = -16 * a.vote_rho, c = 16 * a.lambda_x + 2;
    // band changes of the R rows of exchange step s: two vote lists a row (entering, leaving), four lists per
    // producer warp, their first 64 votes loaded before the rows are cleared
    auto produce = [&](int s) {
        const int v0 = vmax - 1 - s * R, n = min(R, v0 - vtop + 1), t = tid - 32 * P.warps;
        int *half = S.ring + (s & 1) * R * stride;
        constexpr int kLists = 2 * kMaxRows / kProducers;
        int src[kLists], col[kLists][2];
        // the literal bottom band has other lists, but only on the rows down to vmax - chi - 1
        const bool plain = !a.band_literal || v0 < vmax - a.chi - 1;
#pragma unroll
        for (int i = 0; i < kLists; ++i) {
            const int l = warp - P.warps + i * kProducers, v = v0 - (l >> 1);
            const int r = (l & 1) ? v + a.chi + 1 : v - a.chi;
            src[i] = plain && l < 2 * n && r >= vtop && r <= vmax ? r : -1;
            const int m = src[i] >= 0 ? S.cnt[src[i]] : 0;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                col[i][h] = lane + 32 * h < m ? (int)__ldg(vote_list(a, f, src[i]) + lane + 32 * h) : -1;
        }
        {
            constexpr uint32_t kStep = 16 * 32 * kProducers;
            uint32_t z = sa(half) + 16u * (uint32_t)t;
            const uint32_t end = sa(half) + 4u * (uint32_t)(n * stride);
            for (; z + 5 * kStep < end; z += 6 * kStep)
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    sts4(z + k * kStep, make_int4(0, 0, 0, 0));
            for (; z < end; z += kStep)
                sts4(z, make_int4(0, 0, 0, 0));
        }
        // (barrier.sync, not bar.sync, which wants a converged warp: the loops above end per lane)
        asm volatile("barrier.sync 1, %0;" ::"n"(32 * kProducers) : "memory");
        if (plain) {
#pragma unroll
            for (int i = 0; i < kLists; ++i) {
                if (src[i] < 0)
                    continue;
                const int l = warp - P.warps + i * kProducers, by = (l & 1) ? -scale : scale;
                const uint32_t to = sa(half + (l >> 1) * stride + HC);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (col[i][h] >= 0 && LD_IN(col[i][h], W, CK_VPX_VOTE))
                        atoms_add(to + 4u * (uint32_t)col[i][h], by);
                if (S.cnt[src[i]] > 64)
                    add_votes(a, S, f, src[i], 64, to, by, lane, 32);
            }
        } else {
            for (int r = 0; r < n; ++r)
                scatter_delta(a, S, f, v0 - r, vtop, sa(half + r * stride + HC), scale, t, 32 * kProducers);
        }
    };
    // counts of row vmax (the votes of rows [max(vtop, vmax - chi), vmax]) in the first row of the second half
    int *row0 = S.ring + R * stride;
    for (int i = tid; i < stride; i += nt)
        row0[i] = 0;
    __syncthreads();
    // (the literal bottom band of row vmax is [vmax, vmax])
    for (int r = (a.band_literal ? vmax : max(vtop, vmax - a.chi)) + warp; r <= vmax; r += nt >> 5)
        add_votes(a, S, f, r, 0, sa(row0 + HC), scale, lane, 32);
    __syncthreads();
    const int u0 = warp * P.own - HC + lane * C;      // first cell of the lane
    const int cell = warp * P.own + lane * C;         // and its index in a ring row
    const int plane = bt_plane(W, C);
    const bool own = dp && lane >= HL && lane < 32 - HL && u0 < W;
    DpRow<TAU, C> D;
    int nb[C];                                        // the cells' keys of the band, -16 varrho m
    // backtrack bytes of the lane's cells: the ranks in the low bits of `key`, and which cells hold votes
    auto store = [&](uint8_t *out, const int *key) {
#pragma unroll
        for (int x = 0; x < C; x += 4) {
            const uint32_t r = __byte_perm(__byte_perm(key[x], key[x + 1], 0x0040), __byte_perm(key[x + 2], key[x + 3], 0x0040), 0x5410);
            const uint32_t m = __byte_perm(__byte_perm(nb[x], nb[x + 1], 0x0073), __byte_perm(nb[x + 2], nb[x + 3], 0x0073), 0x5410);
            if (own)
                *reinterpret_cast<uint32_t *>(out + x / 4 * plane) = (r & 0x0f0f0f0fu) | (m & (kHasVotes * 0x01010101u));
        }
    };
    if (dp) {
#pragma unroll
        for (int x = 0; x < C; ++x) {
            const bool in = u0 + x >= 0 && u0 + x < W;
            nb[x] = in ? row0[cell + x] : kOffRow;
            D.f[x] = in ? nb[x] : kOffKey;
        }
        store(gbt + (size_t)vmax * RB + 4 * (u0 / C), D.f);   // the last row: no step, but its votes
        if (a.dbg_mx && own)
            for (int x = 0; x < C; ++x)
                if (u0 + x < W)
                    a.dbg_mx[((size_t)f * a.H + vmax) * W + u0 + x] = nb[x] / 16;
    } else {
        produce(0);
    }
    __syncthreads();
    const int steps = (vmax - vtop + R - 1) / R;
    [[maybe_unused]] int low = 0;                     // lowest key at an exchange
    for (int s = 0; s < steps; ++s) {
        const uint32_t box = sa(S.box + (s & 1) * P.warps * 2 * HC);   // [warps][2][HC]
        if (dp) {
            const int vhi = vmax - 1 - s * R, n = min(R, vhi - vtop + 1);
            uint32_t delta = sa(S.ring + (s & 1) * R * stride + cell);
            uint8_t *out = gbt + (size_t)vhi * RB + 4 * (u0 / C);
            int4 d[C / 4];                          // band changes of the next row
#pragma unroll
            for (int x = 0; x < C / 4; ++x)
                d[x] = lds4(delta + 16 * x);
            D.edges(c);
            // one basic block a row, so that a row's packing and stores overlap its shuffles
            auto rows = [&](auto capture) {
                constexpr int kUnroll = decltype(capture)::value ? 1 : 2;   // (less to compile where time matters less)
#pragma unroll kUnroll
                for (int r = 0; r < n; ++r) {
#pragma unroll
                    for (int x = 0; x < C / 4; ++x) {
                        nb[4 * x] += d[x].x;
                        nb[4 * x + 1] += d[x].y;
                        nb[4 * x + 2] += d[x].z;
                        nb[4 * x + 3] += d[x].w;
                    }
                    delta += 4u * (uint32_t)stride;
#pragma unroll
                    for (int x = 0; x < C / 4; ++x)
                        d[x] = lds4(delta + 16 * x);
                    int best[C];
                    D.minima(c, best);
#pragma unroll
                    for (int x = 0; x < C; ++x)
                        D.f[x] = (best[x] & ~15) + nb[x];
                    D.edges(c);
                    store(out, best);
                    out -= RB;
                    if (decltype(capture)::value && own && a.dbg_mx)
                        for (int x = 0; x < C; ++x)
                            if (u0 + x < W)
                                a.dbg_mx[((size_t)f * a.H + vhi - r) * W + u0 + x] = nb[x] / 16;
                }
            };
            if (LOOK || a.dbg_mx)
                rows(std::true_type());
            else
                rows(std::false_type());
            if constexpr (LOOK)
#pragma unroll
                for (int x = 0; x < C; ++x) {
                    low = min(low, D.f[x]);
                    D.f[x] = max(D.f[x], kKeyFloor);
                }
            if (s + 1 < steps) {
                // edge cells the neighbours need: a warp's first owned lanes, and its last
                auto put = [&](int side, int l0) {
                    if (lane >= l0 && lane < l0 + HL)
#pragma unroll
                        for (int x = 0; x < C; x += 4)
                            sts4(box + 4u * (uint32_t)((warp * 2 + side) * HC + (lane - l0) * C + x),
                                 make_int4(D.f[x], D.f[x + 1], D.f[x + 2], D.f[x + 3]));
                };
                put(0, HL);
                put(1, 32 - 2 * HL);
            }
        } else if (s + 1 < steps) {
            produce(s + 1);
        }
        __syncthreads();
        if (dp && s + 1 < steps) {
            const bool lower = lane < HL && warp > 0, upper = lane >= 32 - HL && warp + 1 < P.warps;
            const uint32_t from = box + 4u * (uint32_t)(lower ? ((warp - 1) * 2 + 1) * HC + lane * C
                                                              : (warp + 1) * 2 * HC + (lane - (32 - HL)) * C);
            if (lower || upper)
#pragma unroll
                for (int x = 0; x < C; x += 4) {
                    const int4 e = lds4(from + 4 * x);
                    D.f[x] = e.x;
                    D.f[x + 1] = e.y;
                    D.f[x + 2] = e.z;
                    D.f[x + 3] = e.w;
                }
        }
    }
    if constexpr (LOOK)
        if (__syncthreads_or(low < kKeyFloor))
            return -1;
    int bv = 0x7fffffff, bi = 0x7fffffff;
    if (own)
#pragma unroll
        for (int x = 0; x < C; ++x)
            if (u0 + x < W && D.f[x] < bv) {
                bv = D.f[x];
                bi = u0 + x;
            }
    return block_argmin(bv, bi, S.sh + kMaxChunks);
}

// A function of its own for the frames that need the look: as a branch in the others' loop it cost them 2 % of the
// kernel (64 frames of 1242 x 375: 100.4 us, 98.3 without), as an early end of the loop 6 %.
template <int TAU, int C>
__device__ __noinline__ int vpx_forward_look(const VpxArgs a, const VpxMem S, const VpxPlan P, int f, int vtop, uint8_t *gbt)
{
    return vpx_forward<TAU, C, true>(a, S, P, f, vtop, gbt);
}

// The same with plain energies, for a frame whose best path gathers more than 2^26 - 2^16 (67 million; 1242 x 375 pixels
// with the default parameters cannot hold that much, 1920 x 1080 only if two thirds of all pixels vote for the path's
// columns): rows in shared memory (five of the ring's), compare-select in tie order, a barrier a row, after the packed form
// in vain.  A frame of 120 x 1088 whose votes all converge: 1.43 ms in all (1.63 with a run-time tau_x and two barriers a
// row), 0.37 when its keys fit.
template <int TAU>
__device__ __noinline__ int vpx_forward_wide(const VpxArgs a, const VpxMem S, const VpxPlan P, int f, int vtop, uint8_t *gbt)
{
    const int W = a.W, vmax = a.H - 1, RB = bt_row(W, P.cells), lambda = a.lambda_x;
    const int tid = threadIdx.x, nt = blockDim.x, HC = P.halo * P.cells;
    const int plane = bt_plane(W, P.cells);
    int *Ep = S.ring + HC, *Ec = Ep + P.stride, *band = Ec + P.stride, *delta = band + P.stride;   // delta: two rows in turn
    for (int u = tid; u < W; u += nt)
        band[u] = delta[u] = delta[P.stride + u] = 0;
    __syncthreads();
    const int r0 = a.band_literal ? vmax : max(vtop, vmax - a.chi);
    for (int r = r0; r <= vmax; ++r)
        add_votes(a, S, f, r, 0, sa(band), 1, tid, nt);
    if (vmax > vtop)
        scatter_delta(a, S, f, vmax - 1, vtop, sa(delta + ((vmax - 1) & 1) * P.stride), 1, tid, nt);
    __syncthreads();
    for (int u = tid; u < W; u += nt) {
        Ep[u] = -a.vote_rho * band[u];
        gbt[(size_t)vmax * RB + bt_byte(u, P.cells, plane)] = band[u] ? (uint8_t)kHasVotes : (uint8_t)0;
        if (a.dbg_mx)
            a.dbg_mx[((size_t)f * a.H + vmax) * W + u] = Ep[u];
    }
    __syncthreads();
    for (int v = vmax - 1; v >= vtop; --v) {
        if (v > vtop)   // the next row's changes, while this row is formed
            scatter_delta(a, S, f, v - 1, vtop, sa(delta + ((v - 1) & 1) * P.stride), 1, tid, nt);
        int *dv = delta + (v & 1) * P.stride;
        uint8_t *row = gbt + (size_t)v * RB;
        for (int u = tid; u < W; u += nt) {
            int best = Ep[u], arg = 0;
#pragma unroll
            for (int k = 1; k <= 2 * TAU; ++k) {
                const int d = (k + 1) >> 1, t = (k & 1) ? -d : d;
                if (u + t < 0 || u + t >= W)
                    continue;
                const int cand = Ep[u + t] + lambda * d;
                arg = cand < best ? k : arg;
                best = min(cand, best);
            }
            const int m = band[u] + dv[u];
            band[u] = m;
            dv[u] = 0;
            Ec[u] = best - a.vote_rho * m;
            row[bt_byte(u, P.cells, plane)] = (uint8_t)(arg | (m ? kHasVotes : 0u));
            if (a.dbg_mx)
                a.dbg_mx[((size_t)f * a.H + v) * W + u] = -a.vote_rho * m;
        }
        __syncthreads();
        int *t = Ep;
        Ep = Ec;
        Ec = t;
    }
    int bv = 0x7fffffff, bi = 0x7fffffff;
    for (int u = tid; u < W; u += nt)
        if (Ep[u] < bv) {
            bv = Ep[u];
            bi = u;
        }
    return block_argmin(bv, bi, S.sh + kMaxChunks);
}

template <int TAU, int C>
__device__ __forceinline__ void vpx_dp_body(const VpxArgs &a, const VpxPlan &P, const int f)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int W = a.W, H = a.H, RB = bt_row(W, C);
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const FrameState fs0 = a.fs[f];
    if (fs0.flags & LD_F_NO_LANES)
        return;
    const int vtop = fs0.v_top, vmax = H - 1;
    if (!LD_IN(vtop, H, CK_VPX_TILE) || !LD_IN(W - 1, P.warps * P.own, CK_VPX_TILE))
        return;

    VpxMem S;
    unsigned char *p = smem;
    S.cnt = carve<int16_t>(p, H);
    S.path = carve<int16_t>(p, H);
    S.sup = carve<uint8_t>(p, H);
    S.sh = carve<int>(p, kMaxChunks + 64);
    S.pid = carve<int16_t>(p, H);
    S.box = carve<int>(p, (size_t)2 * P.warps * 2 * P.halo * C);
    S.ring = carve<int>(p, 0);
    uint8_t *gbt = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(a.M1 + (size_t)f * H * W) + 15) & ~(uintptr_t)15);

    // ---- votes per row of [vtop, vmax], and their total ----
    int votes = 0;
    for (int v = tid; v < H; v += nt) {
        int c = v >= vtop ? a.vcount[(size_t)f * H + v] : 0;
        c = LD_IN(c, W + 1, CK_VPX_VOFF) ? c : 0;   // a row holds at most W votes
        S.cnt[v] = (int16_t)c;
        votes += c;
    }
    votes = __reduce_add_sync(0xffffffffu, votes);
    if (lane == 0)
        S.sh[warp] = votes;
    __syncthreads();
    votes = 0;
    for (int k = 0; k < nw; ++k)
        votes += S.sh[k];
    const bool look = 16.0 * a.vote_rho * (2.0 * a.chi + 1.0) * votes >= 2147483648.0 - 1048576.0;
    int ustar = look ? vpx_forward_look<TAU, C>(a, S, P, f, vtop, gbt) : vpx_forward<TAU, C, false>(a, S, P, f, vtop, gbt);
    if (ustar < 0)
        ustar = vpx_forward_wide<TAU>(a, S, P, f, vtop, gbt);

    // ---- backtrack from (ustar, vtop): blocks of kBlock rows.  While lane 0 of warp 0 walks a block, the other
    // warps fetch the columns the next one can reach (2 kBlock rows of tau_x from the current column) and turn
    // their ranks into displacements.
    constexpr int kReach = 2 * kBlock * TAU;
    constexpr int kSlots = (2 * kReach / C + 2 + 3 + 3) / 4 * 4;   // slots of a window: kReach columns on either side
    constexpr int kWinRow = kSlots * C;
    int8_t *win = reinterpret_cast<int8_t *>(S.ring);      // [2][kBlock][kWinRow]
    // window of the block at row lo around column u, from slot max(0, u - kReach) / C / 4 * 4 on: a warp per
    // row, four slots' words of a plane per lane (warps [w0, nw) take part)
    auto first_slot = [&](int u) { return max(u - kReach, 0) / C & ~3; };
    const int plane = bt_plane(W, C);
    auto fetch = [&](int lo, int u, int w0) {
        const int s0 = first_slot(u), quads = min(kSlots / 4, plane / 16 - s0 / 4), n = min(kBlock, vmax - lo);
        const uint32_t to = sa(win) + (uint32_t)(((lo - vtop) / kBlock & 1) * kBlock * kWinRow + 4 * lane * C);
        const uint8_t *from = gbt + (size_t)lo * RB + 4 * s0 + 16 * lane;
        constexpr int kAtOnce = 3;   // rows in flight
        for (int r0 = warp - w0; r0 < n; r0 += kAtOnce * (nw - w0))
            for (int q = 0; q < quads; q += 32) {   // one round unless tau_x is large and C small
                uint4 x[kAtOnce][C / 4];
#pragma unroll
                for (int i = 0; i < kAtOnce; ++i) {
                    const int r = r0 + i * (nw - w0);
#pragma unroll
                    for (int pl = 0; pl < C / 4; ++pl)
                        if (r < n && q + lane < quads)
                            x[i][pl] = __ldcg(reinterpret_cast<const uint4 *>(from + (size_t)r * RB + pl * plane + 16 * q));
                }
                auto steps = [](uint32_t r) { return ((r >> 1) & 0x07070707u) ^ ((r & 0x01010101u) * 0xffu); };   // 0, -1, +1, -2, ...
#pragma unroll
                for (int i = 0; i < kAtOnce; ++i) {
                    const int r = r0 + i * (nw - w0);
                    if (r < n && q + lane < quads)
#pragma unroll
                        for (int pl = 0; pl < C / 4; ++pl) {
                            const uint32_t at = to + (uint32_t)(r * kWinRow + 4 * q * C + 4 * pl);
                            sts1(at, steps(x[i][pl].x));
                            sts1(at + C, steps(x[i][pl].y));
                            sts1(at + 2 * C, steps(x[i][pl].z));
                            sts1(at + 3 * C, steps(x[i][pl].w));
                        }
                }
            }
    };
    int u = ustar, centre = ustar;   // the block's first column, and the column its window lies around
    fetch(vtop, u, 0);
    if (tid == 0)
        S.path[vtop] = (int16_t)u;
    __syncthreads();
    for (int lo = vtop, k = 0; lo < vmax; lo += kBlock, k ^= 1) {
        if (warp > 0) {
            if (lo + kBlock < vmax)
                fetch(lo + kBlock, u, 1);
        } else if (lane == 0) {
            const int hi = min(lo + kBlock, vmax);
            uint32_t at = sa(win + k * kBlock * kWinRow) - (uint32_t)(first_slot(centre) * C);
            int x = u;
#pragma unroll 8
            for (int v = lo; v < hi; ++v, at += kWinRow) {
                if (LD_IN(x, W, CK_VPX_PATH))
                    x += lds_s8(at + (uint32_t)x);
                S.path[v + 1] = (int16_t)x;
            }
            S.sh[k] = x;
        }
        __syncthreads();
        centre = u;
        u = S.sh[k];
    }
    __syncthreads();

    // ---- rows whose path cell holds votes ----
    for (int v = tid; v < H; v += nt)
        S.sup[v] = v >= vtop && LD_IN(S.path[v], W, CK_VPX_PATH)
                       ? (__ldcg(gbt + (size_t)v * RB + bt_byte(S.path[v], C, plane)) & kHasVotes) != 0 : 0;
    __syncthreads();
    const int t = vmax - vtop + 1;
    const int k = block_compact(S.sup + vtop, t, S.pid, S.sh);
    int16_t *gp = a.pts + ((size_t)f * 2 + 1) * 3 * a.pmax;
    for (int j = tid; j < k; j += nt)
        if (LD_IN(j, a.pmax, CK_VPX_PTS) && LD_IN(S.pid[j], t, CK_VPX_PTS)) {
            gp[j] = (int16_t)(vtop + S.pid[j]);
            gp[a.pmax + j] = S.path[vtop + S.pid[j]];
            gp[2 * a.pmax + j] = (int16_t)(vtop + S.pid[j]);
        }
    for (int v = tid; v < H; v += nt)
        a.path_x[(size_t)f * H + v] = v >= vtop ? S.path[v] : (int16_t)0;
    if (tid == 0)
        a.npts[f * 2 + 1] = k;
}

// fd: the frames' descriptors (frame f is fd[f]), or null when the frames share `same`.
template <int TAU, int C, int WARPS>
__global__ void __launch_bounds__(32 * (WARPS + kProducers), 1) k_vpx_dp(const VpxArgs same, const FrameDesc *__restrict__ fd,
                                                                           const VpxPlan P)
{
    VpxArgs a = same;
    if (fd)
        a = vpx_args(fd[blockIdx.x].kp, fd[blockIdx.x].w);
    vpx_dp_body<TAU, C>(a, P, fd ? 0 : blockIdx.x);
}

// Cells per lane: the kernel's instances.
constexpr int kCells[] = {8, 12, kMaxCells};

// The layout of rows of W cells: among the instances and four or eight DP warps, the one whose row is
// estimated fastest.  Measured, a row costs a warp about 25 cycles a cell and 90 more, and an exchange about
// 800 with the loop around it; eight warps share the schedulers in pairs.
VpxPlan vpx_plan(int W, int tau)
{
    VpxPlan best{};
    double best_cost = 1e30;
    for (int C : kCells)
        for (int nw = 4; nw <= (C == kMaxCells ? 8 : 4); nw *= 2) {
            VpxPlan p{};
            p.cells = C;
            p.warps = nw;
            const int lanes = ((W + nw - 1) / nw + C - 1) / C;   // owned lanes a warp needs
            if (lanes > 32)
                continue;
            p.rows = kMaxRows;
            if (tau > 0) {
                const int room = (32 - lanes) / 2 < 10 ? (32 - lanes) / 2 : 10;   // a halo lies within the neighbour's own lanes
                if (room * C < tau)
                    continue;
                p.rows = room * C / tau < kMaxRows ? room * C / tau : kMaxRows;
                p.halo = (tau * p.rows + C - 1) / C;
            }
            p.own = (32 - 2 * p.halo) * C;
            p.stride = nw * p.own + 2 * p.halo * C;
            while (p.rows > 2 && (size_t)(2 * p.rows + 1) * p.stride * sizeof(int) > kRingBytes)
                --p.rows;
            const double cost = (25.0 * C + 90.0 + 800.0 / p.rows) * (nw / 4);
            if (cost < best_cost) {
                best_cost = cost;
                best = p;
            }
        }
    return best;
}

// Shared memory as the kernel carves it: the fixed arrays, then the larger of the ring and the two backtrack
// windows.
size_t vpx_smem(const KParams &kp, const VpxPlan &P)
{
    size_t s = 0;
    auto add = [&](size_t bytes) { s = ((s + 15) & ~(size_t)15) + bytes; };
    add(2 * (size_t)kp.H);
    add(2 * (size_t)kp.H);
    add(kp.H);
    add(4 * (kMaxChunks + 64));
    add(2 * (size_t)kp.H);
    add(4 * (size_t)(2 * P.warps * 2 * P.halo * P.cells));
    s = (s + 15) & ~(size_t)15;
    const size_t ring = (size_t)(2 * (P.rows > 2 ? P.rows : 2) + 1) * P.stride * sizeof(int);
    const size_t windows = (size_t)2 * kBlock * ((4 * kBlock * kp.tau_x / P.cells + 2 + 3 + 3) / 4 * 4) * P.cells;
    return s + (ring > windows ? ring : windows);
}

using VpxKernel = void (*)(VpxArgs, const FrameDesc *, VpxPlan);
template <int TAU>
VpxKernel vpx_kernel_tau(int cells, int warps)
{
    switch (cells) {
    case 8: return k_vpx_dp<TAU, 8, 4>;
    case 12: return k_vpx_dp<TAU, 12, 4>;
    default: return warps == 4 ? k_vpx_dp<TAU, kMaxCells, 4> : k_vpx_dp<TAU, kMaxCells, 8>;
    }
}
VpxKernel vpx_kernel(int tau, int cells, int warps)
{
    switch (tau) {
    case 0: return vpx_kernel_tau<0>(cells, warps);
    case 1: return vpx_kernel_tau<1>(cells, warps);
    case 2: return vpx_kernel_tau<2>(cells, warps);
    case 3: return vpx_kernel_tau<3>(cells, warps);
    case 4: return vpx_kernel_tau<4>(cells, warps);
    case 5: return vpx_kernel_tau<5>(cells, warps);
    case 6: return vpx_kernel_tau<6>(cells, warps);
    default: return vpx_kernel_tau<7>(cells, warps);
    }
}
cudaError_t launch(const KParams &shape, const VpxArgs &a, const FrameDesc *fd, int n, cudaStream_t s)
{
    const VpxPlan P = vpx_plan(shape.W, shape.tau_x);
    vpx_kernel(shape.tau_x, P.cells, P.warps)<<<n, 32 * (P.warps + kProducers), vpx_smem(shape, P), s>>>(a, fd, P);
    return cudaGetLastError();
}

}  // namespace

// Frames a handle accepts: a limit on the frame size and the band height that is part of ld_create's contract (it is what a
// kernel with the votes staged and column bitmaps of the band in shared memory needs: four rows of cells, 12288 votes,
// the per-row arrays, then the bitmaps).  k_vpx_dp needs less: the ring of any layout is at most kRingBytes or five rows,
// beside it are 7 H bytes, the edge cells and the backtrack's block list.
bool vpx_admits(const KParams &kp, size_t budget)
{
    const size_t H = kp.H, cells = (size_t)(kp.W + 1) / 2 * 2;
    size_t s = 0;
    auto add = [&](size_t bytes) { s = ((s + 15) & ~(size_t)15) + bytes; };
    add(4 * (cells + 32));
    add(4 * (cells + 32));
    add(4 * cells);
    add(4 * cells);
    add(4 * (H + 1));
    add(2 * 12288);
    add(2 * H);
    add(H);
    add(4 * (kMaxChunks + 64));
    add(2 * H);
    add(16 * H);
    const size_t fixed = ((s + 15) & ~(size_t)15) + 64;
    const size_t needed = kRingBytes + 7 * (H + 16) + 4 * (kMaxChunks + 64) + 4 * 2 * 8 * 2 * 10 * kMaxCells;
    return budget > fixed + (size_t)4 * kp.W * ((32 + 2 * kp.chi + 32 + 31) / 32 + 1) && budget > needed;
}

// The instances a handle with this tau_x can launch.
cudaError_t setup_vpx(int smem_optin, int tau)
{
    cudaError_t e = cudaSuccess;
    for (int C : kCells)
        for (int warps = 4; warps <= (C == kMaxCells ? 8 : 4); warps *= 2)
            if (e == cudaSuccess)
                e = allow_max_smem(vpx_kernel(tau, C, warps), smem_optin);
    return e;
}

cudaError_t launch_vpx_fd(const KParams &kmax, const FrameDesc *fd, int n, cudaStream_t s)
{
    return launch(kmax, VpxArgs{}, fd, n, s);
}

cudaError_t launch_vpx(const KParams &kp, const Work &w, cudaStream_t s)
{
    return launch(kp, vpx_args(kp, w), nullptr, kp.n_frames, s);
}

}  // namespace ld
