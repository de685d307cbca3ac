// k_road_dp, one CTA per frame: dynamic programming over the v-disparity map, Sec. 2.2, Eq. 11-12: from
// d = D-1 down to d = 1,
//   E_d(v) = -m_y(d, v) + min_{tau in [0, tau_y], v + tau <= H-1} [E_{d+1}(v + tau) + lambda_y tau],
// backtrack buffer the size of the map (4-bit entries), path M_y = {(d, v_d)}.
//
// Readings: Eq. 12 as printed draws on E(v - tau)_{d+1} with -lambda tau; with rows counted from the top and
// road disparity growing downwards, the consistent form links (d, v) to (d+1, v + tau) with a +lambda tau
// penalty (the printed form is kept as the dp_literal switch, k_road_dp_lit).  Ties take the smaller tau; a
// path starts at the smallest index minimising its last row.  A path point whose cell holds no count carries
// no observation; the kernel hands the points with data to the RANSAC fit (k_fit), in increasing index order.
//
// Each DP step is one row of the map.  A thread owns a pair of adjacent cells (many warps per step: the
// step loops are latency-bound) and writes their two 4-bit backtrack entries as one byte.  A thread loads the window of
// the previous row its cells share once.  The CTA is sized to the row, so the per-row barriers involve few
// warps.  Rows are padded with sentinels so the candidate loops have no bounds checks.
#include "k_dp.cuh"

namespace ld {

namespace {

constexpr int kPadY = 20;          // >= 2 + tau_y (rounded up to even)

// ---------------------------------------------------------------------------------------------------
// k_road_dp
// ---------------------------------------------------------------------------------------------------
template <int TMAX>
__device__ __forceinline__ void road_dp_body(const KParams &kp, const Work &w, const int f)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int H = kp.H, D = kp.D, Hp = (H + 1) >> 1;  // Hp: pairs of rows
    const int tid = threadIdx.x, nt = blockDim.x;
    const int32_t *my = w.myT + (size_t)f * D * H;

    unsigned char *p = smem;
    int *E0 = carve<int>(p, 2 * Hp + kPadY);
    int *E1 = carve<int>(p, 2 * Hp + kPadY);
    int *sh = carve<int>(p, kMaxChunks + 64);
    int16_t *path = carve<int16_t>(p, D);
    uint8_t *flag = carve<uint8_t>(p, D);
    int16_t *pid = carve<int16_t>(p, D);
    uint8_t *bt = carve<uint8_t>(p, (size_t)D * Hp);  // one byte per pair of rows: two 4-bit steps

    // E rows hold keys 16 E: a candidate's key 16 (E + lambda tau) + tau orders candidates by energy, then
    // by the smaller tau, so the tie-broken argmin is a plain integer minimum (|16 E| < 2^30 always holds
    // here: energies are bounded by (w + lambda_y tau_y) D).
    for (int v = tid; v < 2 * Hp + kPadY; v += nt) {
        E0[v] = v < H ? -16 * my[(size_t)(D - 1) * H + v] : kSent;
        E1[v] = kSent;
    }
    // thread i owns rows v0 = 2i, v0 + 1.  The data terms of a step are loaded kSets steps ahead into one of
    // kSets register sets (steps rotate over them), so no register copy waits for a load in flight.
    const int i = tid, v0 = 2 * i;
    const bool own = i < Hp;
    auto load_row = [&](int d, int *dst) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int v = v0 + c;
            dst[c] = (own && d >= 1 && v < H) ? __ldg(my + (size_t)d * H + v) : 0;
        }
    };
    constexpr int kSets = 16;  // steps of load latency hidden: kSets - 1
    int reg[kSets][2];
#pragma unroll
    for (int k = 0; k < kSets; ++k)
        load_row(D - 2 - k, reg[k]);
    __syncthreads();
    int *Ep = E0, *Ec = E1;
    const int tau = kp.tau_y;
    int ck[TMAX + 1];  // key offset of step t; steps beyond tau_y never win
#pragma unroll
    for (int t = 0; t <= TMAX; ++t)
        ck[t] = t <= tau ? 16 * kp.lambda_y * t + t : kSent;
    constexpr int NL = (TMAX + 3) / 2;  // 8-byte loads: rows v0 .. v0 + 1 + TMAX
    auto step = [&](int d, const int *cur) {
        if (own) {
            int e[2 * NL];
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                const int2 v2 = *reinterpret_cast<const int2 *>(Ep + v0 + 2 * j);
                e[2 * j] = v2.x;
                e[2 * j + 1] = v2.y;
            }
            uint32_t code = 0;
            int out[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                int kk[TMAX + 1];
#pragma unroll
                for (int t = 0; t <= TMAX; ++t)
                    kk[t] = e[c + t] + ck[t];
#pragma unroll
                for (int st = 1; st <= TMAX; st *= 2)
#pragma unroll
                    for (int j = 0; j + st <= TMAX; j += 2 * st)
                        kk[j] = min(kk[j], kk[j + st]);
                out[c] = v0 + c < H ? -16 * cur[c] + (kk[0] & ~15) : kSent;
                code |= (uint32_t)(kk[0] & 15) << (4 * c);
            }
            *reinterpret_cast<int2 *>(Ec + v0) = make_int2(out[0], out[1]);
            bt[(size_t)d * Hp + i] = (uint8_t)code;
        }
        __syncthreads();
        int *tmp = Ep;
        Ep = Ec;
        Ec = tmp;
    };
    for (int d = D - 2; d >= 1; d -= kSets) {
#pragma unroll
        for (int k = 0; k < kSets; ++k)
            if (d - k >= 1) {
                step(d - k, reg[k]);
                load_row(d - k - kSets, reg[k]);
            }
    }
    int bv = 0x7fffffff, bi = 0x7fffffff;
    for (int v = tid; v < H; v += nt)
        if (Ep[v] < bv) {
            bv = Ep[v];
            bi = v;
        }
    const int vstar = block_argmin(bv, bi, sh + kMaxChunks);
    if (tid == 0) {
        path[0] = -1;
        int v = vstar;
        path[1] = (int16_t)v;
        const uint8_t *row = bt + Hp;
        for (int d = 1; d <= D - 2; ++d, row += Hp) {
            if (LD_IN(v, H, CK_ROAD_PATH))
                v += (row[v >> 1] >> (4 * (v & 1))) & 15;
            path[d + 1] = (int16_t)v;
        }
    }
    __syncthreads();
    for (int d = tid; d < D; d += nt) {
        flag[d] = d >= 1 && LD_IN(path[d], H, CK_ROAD_PATH) && my[(size_t)d * H + path[d]] > 0;
        w.path_y[(size_t)f * D + d] = path[d];
    }
    __syncthreads();
    const int k = block_compact(flag, D, pid, sh);
    int16_t *gp = w.pts + (size_t)f * 2 * 3 * w.pmax;
    for (int j = tid; j < k; j += nt)
        if (LD_IN(j, w.pmax, CK_ROAD_PTS) && LD_IN(pid[j], D, CK_ROAD_PTS)) {
            gp[j] = path[pid[j]];
            gp[w.pmax + j] = pid[j];
            gp[2 * w.pmax + j] = pid[j];
        }
    if (tid == 0)
        w.npts[f * 2] = k;
}

// One thread per pair of rows: the tallest frame (LD_MAX_H rows) needs (LD_MAX_H + 1) / 2 threads, rounded
// up to whole warps.  The bound is kept tight so that the 16 register sets of the load pipeline fit without
// spilling.
constexpr int kRoadMaxThreads = 640;
static_assert(((LD_MAX_H + 1) / 2 + 31) / 32 * 32 <= kRoadMaxThreads, "road DP: one thread per pair of rows");

template <int TMAX>
__global__ void __launch_bounds__(kRoadMaxThreads) k_road_dp(const KParams kp, const Work w) { road_dp_body<TMAX>(kp, w, blockIdx.x); }
template <int TMAX>
__global__ void __launch_bounds__(kRoadMaxThreads) k_road_dp_fd(const FrameDesc *__restrict__ fd)
{
    const FrameDesc &d = fd[blockIdx.x];
    const KParams kp = d.kp;   // the frame's parameters, loaded once into registers
    const Work w = d.w;
    road_dp_body<TMAX>(kp, w, 0);
}

// ---------------------------------------------------------------------------------------------------
// k_road_dp_lit: Eq. 12 as printed (dp_literal), for A/B against the reading above:
//   E_d(v) = -m_y(d, v) + min_{tau in [0, tau_y], v - tau >= 0} [E_{d+1}(v - tau) - lambda_y tau],
// ties to the smaller tau; the path starts at the smallest v minimising E_1 and steps to v - tau.  Plain
// per-row loops (a thread per pair of rows, 4-bit backtrack entries of the pair in one byte); the same
// shared-memory layout and outputs as k_road_dp.
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ void road_dp_lit_body(const KParams &kp, const Work &w, const int f)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int H = kp.H, D = kp.D, Hp = (H + 1) >> 1;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int32_t *my = w.myT + (size_t)f * D * H;
    unsigned char *p = smem;
    int *Ep = carve<int>(p, 2 * Hp + kPadY);
    int *Ec = carve<int>(p, 2 * Hp + kPadY);
    int *sh = carve<int>(p, kMaxChunks + 64);
    int16_t *path = carve<int16_t>(p, D);
    uint8_t *flag = carve<uint8_t>(p, D);
    int16_t *pid = carve<int16_t>(p, D);
    uint8_t *bt = carve<uint8_t>(p, (size_t)D * Hp);
    for (int v = tid; v < H; v += nt)
        Ep[v] = -my[(size_t)(D - 1) * H + v];
    __syncthreads();
    const int tau = kp.tau_y, lam = kp.lambda_y;
    for (int d = D - 2; d >= 1; --d) {
        for (int i = tid; i < Hp; i += nt) {
            uint32_t code = 0;
            for (int c = 0; c < 2; ++c) {
                const int v = 2 * i + c;
                if (v >= H)
                    break;
                int best = 0x7fffffff, arg = 0;
                for (int t = 0; t <= tau && v - t >= 0; ++t) {
                    const int cand = Ep[v - t] - lam * t;
                    if (cand < best) {
                        best = cand;
                        arg = t;
                    }
                }
                Ec[v] = -my[(size_t)d * H + v] + best;
                code |= (uint32_t)arg << (4 * c);
            }
            bt[(size_t)d * Hp + i] = (uint8_t)code;
        }
        __syncthreads();
        int *tmp = Ep;
        Ep = Ec;
        Ec = tmp;
    }
    int bv = 0x7fffffff, bi = 0x7fffffff;
    for (int v = tid; v < H; v += nt)
        if (Ep[v] < bv) {
            bv = Ep[v];
            bi = v;
        }
    const int vstar = block_argmin(bv, bi, sh + kMaxChunks);
    if (tid == 0) {
        path[0] = -1;
        int v = vstar;
        path[1] = (int16_t)v;
        for (int d = 1; d <= D - 2; ++d) {
            if (LD_IN(v, H, CK_ROAD_PATH))
                v -= (bt[(size_t)d * Hp + (v >> 1)] >> (4 * (v & 1))) & 15;
            path[d + 1] = (int16_t)v;
        }
    }
    __syncthreads();
    for (int d = tid; d < D; d += nt) {
        flag[d] = d >= 1 && LD_IN(path[d], H, CK_ROAD_PATH) && my[(size_t)d * H + path[d]] > 0;
        w.path_y[(size_t)f * D + d] = path[d];
    }
    __syncthreads();
    const int k = block_compact(flag, D, pid, sh);
    int16_t *gp = w.pts + (size_t)f * 2 * 3 * w.pmax;
    for (int j = tid; j < k; j += nt)
        if (LD_IN(j, w.pmax, CK_ROAD_PTS) && LD_IN(pid[j], D, CK_ROAD_PTS)) {
            gp[j] = path[pid[j]];
            gp[w.pmax + j] = pid[j];
            gp[2 * w.pmax + j] = pid[j];
        }
    if (tid == 0)
        w.npts[f * 2] = k;
}

__global__ void __launch_bounds__(1024) k_road_dp_lit(const KParams kp, const Work w) { road_dp_lit_body(kp, w, blockIdx.x); }
__global__ void __launch_bounds__(1024) k_road_dp_lit_fd(const FrameDesc *__restrict__ fd)
{
    const FrameDesc &d = fd[blockIdx.x];
    const KParams kp = d.kp;   // the frame's parameters, loaded once into registers
    const Work w = d.w;
    road_dp_lit_body(kp, w, 0);
}

using RoadKernel = void (*)(KParams, Work);
RoadKernel road_kernel(int tau) { return tau <= 6 ? k_road_dp<6> : k_road_dp<15>; }

}  // namespace

size_t road_smem_bytes(const KParams &kp)
{
    const size_t H = kp.H, D = kp.D, Hp = (H + 1) / 2;
    size_t s = 0;
    auto add = [&](size_t bytes) { s = ((s + 15) & ~(size_t)15) + bytes; };
    add(4 * (2 * Hp + kPadY));
    add(4 * (2 * Hp + kPadY));
    add(4 * (kMaxChunks + 64));
    add(2 * D);
    add(D);
    add(2 * D);
    add(D * Hp);
    return s + 64;
}

// One thread per pair of rows (at least two warps).
int road_threads(int H)
{
    const int nt = ((H + 1) / 2 + 31) / 32 * 32;
    return nt < 64 ? 64 : nt;
}

cudaError_t setup_dp(int smem_optin)
{
    cudaError_t e = allow_max_smem(k_road_dp<6>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_road_dp_lit, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_road_dp<15>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_road_dp_fd<6>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_road_dp_fd<15>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_road_dp_lit_fd, smem_optin);
    return e;
}

cudaError_t launch_road(const KParams &kp, const Work &w, cudaStream_t s)
{
    if (kp.dp_literal)
        k_road_dp_lit<<<kp.n_frames, road_threads(kp.H), road_smem_bytes(kp), s>>>(kp, w);
    else
        road_kernel(kp.tau_y)<<<kp.n_frames, road_threads(kp.H), road_smem_bytes(kp), s>>>(kp, w);
    return cudaGetLastError();
}

cudaError_t launch_road_fd(const KParams &kmax, const FrameDesc *fd, int n, cudaStream_t s)
{
    if (kmax.dp_literal)
        k_road_dp_lit_fd<<<n, road_threads(kmax.H), road_smem_bytes(kmax), s>>>(fd);
    else if (kmax.tau_y <= 6)
        k_road_dp_fd<6><<<n, road_threads(kmax.H), road_smem_bytes(kmax), s>>>(fd);
    else
        k_road_dp_fd<15><<<n, road_threads(kmax.H), road_smem_bytes(kmax), s>>>(fd);
    return cudaGetLastError();
}

}  // namespace ld
