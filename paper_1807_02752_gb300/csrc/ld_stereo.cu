// Stereo matching (Sec. 2.1), the stage that makes the disparity map the lane path takes as input:
// NCC block matching (Eq. 1-8) with search range propagation (Eq. 9, Alg. 2) for the left and the right
// disparity map, then the left-right consistency check (Alg. 3).  Kernels and the ld_stereo_* entry
// points of include/ld.h.
//
//   k_srp   one CTA, or one cluster of CTAs that share a row, per (frame, map): rows from H-1-rho up to rho,
//           in order, since a row's search range comes from the row below (the layout is described at the
//           kernel).  The best candidate has the largest NCC, compared exactly: c = N / sqrt(D_a D_b) with
//           N = n P - s_a s_b and D = n Q - s^2 (s, Q, P: block sums of I, I^2 and the product, exact
//           integers, the quantities the paper gets from integral images, Eq. 5), so
//           c1 > c2 <=> N1 |N1| D2 > N2 |N2| D1 (a float filter decides clear cases, 128-bit integers the
//           rest).
//   k_lrc   l(u, v) = l_lf(u, v) when |l_lf(u, v) - l_rt(u - l_lf(u, v), v)| <= tr, else 0; float output.
//
// Readings: blocks lie inside both images (other pixels and candidates are skipped; a pixel without a
// candidate gets 0); ties go to the smaller disparity; the first row searches [0, d_max], every later
// pixel the union of [l - tau, l + tau] over the three estimates of the row below that exist.
#include <cstring>
#include <string>

#include "ld_net.cuh"

namespace ld {

namespace {

struct SrpArgs {
    const uint8_t *left, *right;     // [n][H][W]
    int16_t *lf, *rt;                // [n][H][W]
    int W, H, dmax, tau;
    // launch shape (SrpShape)
    int per;                         // pixels a CTA of the cluster owns
    int strips, n_extra;             // its strips, and those of the other image beyond them
    int groups;                      // warps that search a strip (the first strips x groups warps of a CTA)
};

constexpr int kSrpMaxWarps = 24;     // warps of a CTA (80 registers a thread)
constexpr int kSrpFewWarps = 16;     // ... of the variant with 128 registers, for the CTAs of few pairs
constexpr int kSrpPrep = 4;          // strips of the other image a preparing warp takes at most
constexpr int kSrpShared = 12;       // distinct disparities up to which a strip walks their union in any case
constexpr int kSrpHalo = 8;          // rows between two exchanges of a cluster = halo pixels on each side

// Pixels of a strip: a warp's 64 columns less the 2 rho that only complete the blocks of its neighbours.
__host__ __device__ constexpr int srp_strip(int rho) { return 64 - 2 * rho; }
// Entries of one buffer of the other image (16 bytes each).
__host__ __device__ inline int srp_entries(int warps, int n_extra, int rho)
{
    return srp_strip(rho) * (warps + n_extra) + 2 * rho;
}

__device__ __forceinline__ uint32_t srp_shl(uint32_t x, int n)   // 0 for n >= 32
{
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
// Bits b of [0, 32) with lo <= b <= hi.
__device__ __forceinline__ uint32_t srp_bits(int lo, int hi)
{
    return srp_shl(0xffffffffu, max(lo, 0)) & ~srp_shl(0xffffffffu, max(hi + 1, 0));
}
__device__ __forceinline__ float srp_rsqrt(float x)   // x >= 1; relative error at most 2^-22.9
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ uint4 srp_lds(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 srp_lds2(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
// Not the .aligned forms: those want a converged warp, and the exchange calls this right after stores that only
// some lanes make.
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// A lane's two adjacent image columns: the K rows of the block window in K bytes (the newest in byte 0) and
// the window's sums of I and I^2.
template <int RHO>
struct SrpCols {
    uint32_t lo[2], hi[2];
    int s[2], q[2];
    __device__ __forceinline__ void push(int c, int x)   // the row above enters, the bottom row leaves
    {
        constexpr int K = 2 * RHO + 1;
        int old;
        if constexpr (K > 4) {
            old = (int)(hi[c] >> (8 * (K - 5)));
            hi[c] = __funnelshift_l(lo[c], hi[c], 8) & ((1u << (8 * (K - 4))) - 1u);
            lo[c] = (lo[c] << 8) | (uint32_t)x;
        } else {
            old = (int)(lo[c] >> (8 * (K - 1)));
            lo[c] = ((lo[c] << 8) | (uint32_t)x) & ((1u << (8 * K)) - 1u);
        }
        s[c] += x - old;
        q[c] += (x - old) * (x + old);
    }
};

// Sums over the K columns of the blocks of a lane's two pixels (leftmost columns 2 lane and 2 lane + 1 of
// the strip), for N quantities at once, from the per-column values c0, c1: sum_1 = c1 + sum_{k = 1 .. rho}
// (c0 + c1) of lane + k, and sum_0 differs by the outer columns.  Valid on lanes below srp_strip / 2.  The N
// chains go through each shuffle together (shuffles keep their order, so one chain after the other would
// wait out every latency).
template <int RHO, int N>
__device__ __forceinline__ void srp_block_sums(const int *c0, const int *c1, int *p0, int *p1)
{
    constexpr unsigned kAll = 0xffffffffu;
    int t1[N], last[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
        t1[k] = __shfl_down_sync(kAll, c0[k] + c1[k], 1);
#pragma unroll
    for (int k = 0; k < N; ++k)
        last[k] = __shfl_down_sync(kAll, c1[k], RHO);
#pragma unroll
    for (int k = 0; k < N; ++k) {
        if constexpr (RHO == 1)
            p1[k] = c1[k] + t1[k];
        else if constexpr (RHO == 2)
            p1[k] = c1[k] + t1[k] + __shfl_down_sync(kAll, c0[k] + c1[k], 2);
        else
            p1[k] = c1[k] + t1[k] + __shfl_down_sync(kAll, c0[k] + c1[k] + t1[k], 2);
    }
#pragma unroll
    for (int k = 0; k < N; ++k)
        p0[k] = p1[k] + c0[k] - last[k];
}

// Exact comparison, for a pixel whose two best float scores are too close: candidates are the d <= dhi within t of an
// estimate, ascending, in integers N = n P - s_a s_b and D = n Q - s_b^2 from the columns of the other image that the row's
// search used; c1 > c2 <=> N1 |N1| D2 > N2 |N2| D1, and c = 0 where a block is constant (then N = 0).  That is one pixel in
// 10^4 of noise or of a textured pair, but every pixel where an image does not change along its rows or repeats within a
// search range; two candidates of such a pixel have the same N and D, and nothing is multiplied.  The best one so far:
struct SrpBest {
    int d = -1, N = 0, D = 0;
    __device__ __forceinline__ void consider(int d1, int N1, int D1)
    {
        bool better = d < 0;
        if (!better && (N1 != N || D1 != D)) {
            if (N1 == 0 || N == 0)
                better = N1 > N;
            else
                better = (__int128)((long long)N1 * abs(N1)) * D > (__int128)((long long)N * abs(N)) * D1;
        }
        if (better) {
            d = d1;
            N = N1;
            D = D1;
        }
    }
};

// N and D of the block whose columns are (alo, ahi), of sum sa, in image A and the entries from e on in image B.
template <int RHO>
__device__ __forceinline__ void srp_block_nd(const uint32_t *alo, const uint32_t *ahi, int sa, uint32_t buf, uint32_t odd, int e,
                                             int &N, int &D)
{
    constexpr int K = 2 * RHO + 1, NB = K * K;
    const uint32_t at = buf + 16u * (uint32_t)(e >> 1);
    const uint32_t ev = at + ((e & 1) ? odd : 0u), od = at + ((e & 1) ? 16u : odd);
    const uint4 first = srp_lds(ev);
    unsigned P = __dp4a(alo[0], first.x, __dp4a(ahi[0], first.y, 0u));
    unsigned Q = __dp4a(first.x, first.x, __dp4a(first.y, first.y, 0u));
#pragma unroll
    for (int k = 1; k < K; ++k) {
        const uint2 b = srp_lds2((k & 1) ? od + 16u * (uint32_t)(k >> 1) : ev + 16u * (uint32_t)(k >> 1));
        P = __dp4a(alo[k], b.x, __dp4a(ahi[k], b.y, P));
        Q = __dp4a(b.x, b.x, __dp4a(b.y, b.y, Q));
    }
    const int sb = (int)first.z;
    N = NB * (int)P - sa * sb;
    D = NB * (int)Q - sb * sb;
}

// The exact best of pixel (u, v) with the estimates l0, l1, l2, by one lane of a cluster's CTA: the block of A from the
// image, and where the entries lie (k_srp's layout) worked out again, so that k_srp keeps nothing for it.  One pair of
// 1242 x 375 that is constant along its rows: 0.95 ms (1.76 with the blocks of both images summed for each candidate).
template <int RHO>
__device__ __noinline__ int srp_exact_best(const SrpArgs &a, int v, int u, int l0, int l1, int l2, int t, int dhi)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int W = a.W, dir = blockIdx.z, rank = blockIdx.x, sign = dir == 0 ? -1 : 1, S = srp_strip(RHO);
    const uint8_t *block = (dir == 0 ? a.left : a.right) + ((size_t)blockIdx.y * a.H + v - RHO) * W + u - RHO;
    const int col0 = rank * a.per - (rank > 0 ? kSrpHalo : 0), ent0 = col0 - (dir == 0 ? S * a.n_extra : 0);
    const uint32_t odd = 16u * (uint32_t)(srp_entries(a.strips, a.n_extra, RHO) >> 1);
    const uint32_t buf = (uint32_t)__cvta_generic_to_shared(sm) + (uint32_t)(v & 1) * 2u * odd;
    const int e0 = u - RHO - ent0;
    constexpr int K = 2 * RHO + 1;
    uint32_t lo[K], hi[K];   // the block's columns, the top row in byte 0
    unsigned sa = 0;
#pragma unroll
    for (int x = 0; x < K; ++x) {
        lo[x] = hi[x] = 0u;
#pragma unroll
        for (int y = 0; y < K; ++y)
            (y < 4 ? lo : hi)[x] |= (uint32_t)__ldg(block + (size_t)y * W + x) << (8 * (y & 3));
        sa = __dp4a(lo[x], 0x01010101u, __dp4a(hi[x], 0x01010101u, sa));
    }
    SrpBest best;
    for (int d = max(min(min(l0, l1), l2) - t, 0); d <= min(max(max(l0, l1), l2) + t, dhi); ++d)
        if (abs(d - l0) <= t || abs(d - l1) <= t || abs(d - l2) <= t) {
            int N, D;
            srp_block_nd<RHO>(lo, hi, (int)sa, buf, odd, e0 + sign * d, N, D);
            best.consider(d, N, D);
        }
    return best.d;
}

// The lane's two columns and its right neighbours': the K + 1 columns of the blocks of a lane's two pixels.
template <int RHO>
__device__ __forceinline__ void srp_columns(const uint32_t (&lo)[2], const uint32_t (&hi)[2], uint32_t (&clo)[2 * RHO + 2],
                                            uint32_t (&chi)[2 * RHO + 2])
{
#pragma unroll
    for (int x = 0; x <= RHO; ++x)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            clo[2 * x + c] = __shfl_down_sync(0xffffffffu, lo[c], x);
            chi[2 * x + c] = __shfl_down_sync(0xffffffffu, hi[c], x);
        }
}

// What a warp's exact comparison needs of a row.
struct SrpRow {
    uint32_t buf, odd;                   // shared address of the row's entries, offset of the odd columns
    int q, dir, t;                       // entry of the first pixel's leftmost column at d = 0
    int sa[2], dhi[2], l[2][3], d[2];    // the lane's two pixels: block sums of A, ranges, the float scores' choice
    bool close[2];                       // too close to call
};

// The same for the pixels of a warp together, the blocks of A from its lanes' registers.  64 pairs that are constant along
// their rows: 1.90 ms (4.96 with the blocks of both images summed for each candidate).
template <int RHO>
__device__ __noinline__ int2 srp_settle(uint32_t lo0, uint32_t lo1, uint32_t hi0, uint32_t hi1, const SrpRow &r)
{
    constexpr int K = 2 * RHO + 1;
    uint32_t alo[K + 1], ahi[K + 1];
    const uint32_t lo[2] = {lo0, lo1}, hi[2] = {hi0, hi1};
    srp_columns<RHO>(lo, hi, alo, ahi);
    int out[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        out[p] = r.d[p];
        if (!r.close[p])
            continue;
        const int l0 = r.l[p][0], l1 = r.l[p][1], l2 = r.l[p][2];
        SrpBest best;
        for (int d = max(min(min(l0, l1), l2) - r.t, 0); d <= min(max(max(l0, l1), l2) + r.t, r.dhi[p]); ++d) {
            if (abs(d - l0) > r.t && abs(d - l1) > r.t && abs(d - l2) > r.t)
                continue;
            int N, D;
            srp_block_nd<RHO>(alo + p, ahi + p, r.sa[p], r.buf, r.odd, r.q + p + (r.dir == 0 ? -d : d), N, D);
            best.consider(d, N, D);
        }
        out[p] = best.d;
    }
    return make_int2(out[0], out[1]);
}

// Layout.  A warp owns a strip of 64 image columns, two adjacent ones per lane, and the 64 - 2 rho pixels
// whose blocks they complete.  Column dot products (two dp4a) of the strip with the other image at one
// disparity d give the block products P of all its pixels through three shuffles, instead of 2 rho + 1
// column products per pixel and candidate: neighbouring pixels mostly search the same few disparities (the
// rows of the synthetic pairs need 6 to 10 distinct ones per strip and row, and 3.3 to 3.8 per pixel), so
// the warp walks the union of its pixels' search ranges, 30 disparities at a time as a bit mask, and each
// pixel takes part at its own candidates.  A lane keeps its columns of image A and their sums in registers
// (the window moves up a row by a byte shift) and publishes the same of image B in shared memory, one
// 16-byte entry per column {rows 0-3, rows 4-6, s_B, 1 / sqrt(D_B)}, even and odd columns apart so that a
// warp's loads of any d are contiguous; double-buffered by row, so one barrier per row suffices.
// N and D fit 32 bits (n^2 255^2 < 2^28).  The score N / sqrt(D_B) is a float: the conversions, the product
// and rsqrt.approx (relative error 2^-22.9) err by less than 2^-21 together, so when the best score leads
// the second best by more than 2^-20 (|s1| + |s2|) the best candidate is the exact one; otherwise the pixel's
// candidates are compared again in integers (SrpBest).  Ascending d and a strict comparison give ties to the
// smaller disparity.
//
// Few pairs leave most SMs idle, so a map's columns are then split over a cluster (CLUSTER): each CTA also
// computes kSrpHalo pixels beyond its own on either side, which a pixel per row becomes stale (a row reads
// its neighbours' estimates one pixel away); every kSrpHalo rows the CTAs write their edge estimates into
// the neighbours' shared memory and meet at a cluster barrier.  A CTA then has few strips, and the row is a
// chain of latencies: one or two warps search a strip (two take the even and the odd disparities and merge
// through shared memory) and others prepare the other image, NPREP strips each.  With a whole map per CTA
// the strips' own warps do both.
//
// What bounds it: the rows follow one another (369 at 1242x375).  One CTA per map: the ALU pipe (two cycles
// per integer instruction) and the wait for the strip with the most distinct disparities.  Clusters: the
// latency chain of a row (about 4400 cycles).  At 1242x375, d_max 127: 64 pairs 3.42 -> 1.57 ms, one pair
// 3.19 -> 0.77 to 0.90 ms by its texture, against every pixel forming its own candidates' products with one CTA
// per map.
template <int RHO, int NPREP, bool CLUSTER, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 1) k_srp(const __grid_constant__ SrpArgs a)
{
    constexpr int S = srp_strip(RHO), K = 2 * RHO + 1, NB = K * K;
    constexpr int kWin = 30;          // disparities of one candidate mask
    constexpr int kBatch = CLUSTER ? 2 : 3;   // disparities of the union in flight together
    extern __shared__ __align__(16) unsigned char sm[];
    const int W = a.W, H = a.H, f = blockIdx.y, dir = blockIdx.z, rank = blockIdx.x, nrank = gridDim.x;
    const size_t fo = (size_t)f * H * W;
    const uint8_t *A = (dir == 0 ? a.left : a.right) + fo;   // the image whose map this is
    const uint8_t *B = (dir == 0 ? a.right : a.left) + fo;
    int16_t *out = (dir == 0 ? a.lf : a.rt) + fo;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = a.strips;
    const int n_search = nw * a.groups, group = warp / nw;   // searching warps: strip warp % nw, group warp / nw
    const bool search = !CLUSTER || warp < n_search;
    const int strip = warp - group * nw;
    const int vb = H - 1 - RHO, umax = W - 1 - RHO;
    const int own0 = RHO + rank * a.per, own1 = min(own0 + a.per, W - RHO);   // pixels [own0, own1)
    const int px0 = own0 - (CLUSTER && rank > 0 ? kSrpHalo : 0);              // first pixel computed
    const int col0 = px0 - RHO;                                               // its leftmost column
    const int ent0 = col0 - (dir == 0 ? S * a.n_extra : 0);                   // column of entry 0
    const int n_ent = srp_entries(nw, a.n_extra, RHO);
    const uint32_t odd = 16u * (uint32_t)(n_ent >> 1), buf_bytes = 2u * odd;
    const uint32_t ent = (uint32_t)__cvta_generic_to_shared(sm);
    // estimates of the row below and of this row: two int16 per pair of pixels, a missing pair before the
    // first and after the last
    uint32_t *lv = reinterpret_cast<uint32_t *>(sm + 2 * (size_t)buf_bytes);   // [2][nw S / 2 + 2]
    const int n_lv = nw * (S / 2) + 2;
    int16_t *inbox = reinterpret_cast<int16_t *>(lv + 2 * n_lv);               // [2][2 kSrpHalo] left, right halo
    float *half = reinterpret_cast<float *>(inbox + 4 * kSrpHalo);             // [6][32 nw] second group's bests

    const int pair = strip * (S / 2) + lane;              // the lane's pair of pixels px0 + 2 pair, + 1
    const int u0 = px0 + 2 * pair;
    const bool mine = lane < S / 2;
    const bool in0 = search && mine && u0 <= umax, in1 = search && mine && u0 + 1 <= umax;
    const bool st0 = in0 && group == 0 && u0 >= own0 && u0 < own1, st1 = in1 && group == 0 && u0 + 1 >= own0 && u0 + 1 < own1;
    int dhi0 = dir == 0 ? u0 - RHO : umax - u0, dhi1 = dir == 0 ? u0 + 1 - RHO : umax - u0 - 1;
    dhi0 = in0 ? min(dhi0, a.dmax) : -1;
    dhi1 = in1 ? min(dhi1, a.dmax) : -1;

    // borders without a block: rows by the first CTA of the cluster, columns likewise
    if (rank == 0) {
        for (int i = tid; i < RHO * W; i += blockDim.x) {
            out[i] = 0;
            out[(size_t)(H - RHO) * W + i] = 0;
        }
        for (int i = tid; i < (H - 2 * RHO) * 2 * RHO; i += blockDim.x) {
            const int r = i / (2 * RHO), c = i - r * 2 * RHO;
            out[(size_t)(RHO + r) * W + (c < RHO ? c : W - 2 * RHO + c)] = 0;
        }
    }
    for (int i = tid; i < 2 * n_lv; i += blockDim.x)
        lv[i] = 0xffffffffu;   // -1: no estimate

    // strips of B this warp prepares (counted from column ent0): its own, or a preparing warp's share
    int bcol[NPREP];
    bool bon[NPREP];
    const int n_prep = (int)(blockDim.x >> 5) - n_search;
#pragma unroll
    for (int k = 0; k < NPREP; ++k) {
        const int at = warp - n_search + k * n_prep;
        bcol[k] = CLUSTER ? ent0 + S * at : col0 + S * strip;
        bon[k] = (CLUSTER ? !search && at < nw + a.n_extra : true) && bcol[k] < W && bcol[k] + 64 > 0;
    }
    const int bend = CLUSTER ? ent0 + S * (nw + a.n_extra) : col0 + S * nw;   // first column no strip begins at
    // row y of the lane's two columns (the caller's pointer to them); columns off the image read 0
    auto load2 = [&](const uint8_t *p, int c, bool on, int *x) {
        x[0] = on && c >= 0 && c < W ? (int)__ldg(p) : 0;
        x[1] = on && c >= -1 && c < W - 1 ? (int)__ldg(p + 1) : 0;
    };
    const int acol = col0 + 2 * pair;
    const uint8_t *pa = A + (ptrdiff_t)(vb + RHO) * W + acol, *pb[NPREP];
#pragma unroll
    for (int k = 0; k < NPREP; ++k)
        pb[k] = B + (ptrdiff_t)(vb + RHO) * W + bcol[k] + 2 * lane;
    SrpCols<RHO> ac = {}, bc[NPREP] = {};
    int sa0 = 0, sa1 = 0;
    auto publish = [&](int k, uint32_t to) {
        const int c0[2] = {bc[k].s[0], bc[k].q[0]}, c1[2] = {bc[k].s[1], bc[k].q[1]};
        int p0[2], p1[2];
        srp_block_sums<RHO, 2>(c0, c1, p0, p1);
        const int s0 = p0[0], q0 = p0[1], s1 = p1[0], q1 = p1[1];
        const int D0 = NB * q0 - s0 * s0, D1 = NB * q1 - s1 * s1;
        const float i0 = D0 > 0 ? srp_rsqrt((float)D0) : 0.0f, i1 = D1 > 0 ? srp_rsqrt((float)D1) : 0.0f;
        const int next = bcol[k] + S;   // the next strip is prepared when it holds columns of the image
        const bool all = next >= W || next >= bend;
        if (mine || all) {
            const uint32_t at = to + 16u * (uint32_t)(((bcol[k] - ent0) >> 1) + lane);
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(bc[k].lo[0]), "r"(bc[k].hi[0]),
                         "r"(s0), "r"(__float_as_int(i0)) : "memory");
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at + odd), "r"(bc[k].lo[1]), "r"(bc[k].hi[1]),
                         "r"(s1), "r"(__float_as_int(i1)) : "memory");
        }
    };
    for (int y = vb + RHO; y >= vb - RHO; --y) {
        int x[2];
        load2(pa, acol, search, x);
        pa -= W;
        ac.push(0, x[0]);
        ac.push(1, x[1]);
#pragma unroll
        for (int k = 0; k < NPREP; ++k) {
            load2(pb[k], bcol[k] + 2 * lane, bon[k], x);
            pb[k] -= W;
            bc[k].push(0, x[0]);
            bc[k].push(1, x[1]);
        }
    }
    srp_block_sums<RHO, 1>(&ac.s[0], &ac.s[1], &sa0, &sa1);
#pragma unroll
    for (int k = 0; k < NPREP; ++k)
        if (bon[k])
            publish(k, ent + (uint32_t)(vb & 1) * buf_bytes);
    // the two rows that enter next, loaded two rows ahead
    int an[2][2], bn[NPREP][2][2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const bool on = vb - RHO - 1 - r >= 0;
        load2(pa, acol, on && search, an[r]);
        pa -= W;
#pragma unroll
        for (int k = 0; k < NPREP; ++k) {
            load2(pb[k], bcol[k] + 2 * lane, on && bon[k], bn[k][r]);
            pb[k] -= W;
        }
    }
    if constexpr (CLUSTER)
        cluster_sync_all();   // every CTA of the cluster has started before its shared memory is written
    else
        __syncthreads();

    const uint32_t jaddr = 16u * (uint32_t)(((col0 - ent0) >> 1) + pair);
    for (int v = vb; v >= RHO; --v) {
        // B of the next row first (the other buffer): it depends on nothing of this row
        if (v > RHO) {
#pragma unroll
            for (int k = 0; k < NPREP; ++k)
                if (bon[k]) {
                    bc[k].push(0, bn[k][0][0]);
                    bc[k].push(1, bn[k][0][1]);
                    publish(k, ent + (uint32_t)((v - 1) & 1) * buf_bytes);
                    bn[k][0][0] = bn[k][1][0];
                    bn[k][0][1] = bn[k][1][1];
                    load2(pb[k], bcol[k] + 2 * lane, v - RHO - 3 >= 0, bn[k][1]);
                    pb[k] -= W;
                }
        }
        int d0 = 0, d1 = 0;
        if (search) {
        // search ranges: [0, dmax] on the first row, else [l - tau, l + tau] around the estimates below of
        // the pixel and its two neighbours (one that is missing repeats the pixel's own)
        int l00 = 0, l01 = 0, l02 = 0, l11 = 0, l12 = 0, t = a.dmax;
        if (v < vb) {
            const uint32_t *below = lv + ((v + 1) & 1) * n_lv + 1;
            const uint32_t wl = mine ? below[pair - 1] : 0u, wc = mine ? below[pair] : 0u, wr = mine ? below[pair + 1] : 0u;
            const int lm = (int)wl >> 16, la = (int)(int16_t)(wc & 0xffffu), lb = (int)wc >> 16,
                      lp = (int)(int16_t)(wr & 0xffffu);
            l01 = la;
            l00 = lm < 0 ? la : lm;
            l02 = lb < 0 ? la : lb;   // the second pixel's range is [l01, l11, l12]
            l11 = lb;
            l12 = lp < 0 ? lb : lp;
            t = a.tau;
        }
        const int mn0 = min(min(l00, l01), l02), mx0 = max(max(l00, l01), l02);
        const int mn1 = min(min(l01, l11), l12), mx1 = max(max(l01, l11), l12);
        int lo = min(in0 ? mn0 : 0x3fffffff, in1 ? mn1 : 0x3fffffff) - t;
        int hi = max(in0 ? min(mx0 + t, dhi0) : -1, in1 ? min(mx1 + t, dhi1) : -1);
        lo = max(__reduce_min_sync(0xffffffffu, lo), 0);
        hi = __reduce_max_sync(0xffffffffu, hi);
        const uint32_t buf = ent + (uint32_t)(v & 1) * buf_bytes;
        const uint32_t lane_ent = buf + jaddr;
        // best and second best score of the two pixels (far below any NCC: none yet) and the best's disparity
        constexpr float kNone = -1e30f;
        float b0 = kNone, b1 = kNone, r0 = kNone, r1 = kNone;
        const int q = (col0 - ent0) + 2 * pair;   // entry of the first pixel's leftmost column at d = 0
        auto consider = [](float s, int d, float &best, float &second, int &dbest) {
            dbest = s > best ? d : dbest;
            second = fmaxf(second, fminf(best, s));
            best = fmaxf(best, s);
        };
        for (int base = lo; base <= hi; base += kWin) {
            // candidates of the two pixels among d = base .. base + kWin - 1
            uint32_t m0, m1;
            if (t == 1) {   // bit k of c: an estimate base - 1 + k, whose range is bits k - 2 .. k of the mask
                const uint32_t cs = srp_shl(1u, l01 - base + 1);
                const uint32_t c0 = cs | srp_shl(1u, l00 - base + 1) | srp_shl(1u, l02 - base + 1);
                const uint32_t c1 = cs | srp_shl(1u, l11 - base + 1) | srp_shl(1u, l12 - base + 1);
                m0 = c0 | (c0 >> 1) | (c0 >> 2);
                m1 = c1 | (c1 >> 1) | (c1 >> 2);
            } else {
                m0 = srp_bits(l00 - t - base, l00 + t - base) | srp_bits(l01 - t - base, l01 + t - base) |
                     srp_bits(l02 - t - base, l02 + t - base);
                m1 = srp_bits(l01 - t - base, l01 + t - base) | srp_bits(l11 - t - base, l11 + t - base) |
                     srp_bits(l12 - t - base, l12 + t - base);
            }
            m0 &= srp_bits(0, min(dhi0 - base, kWin - 1));
            m1 &= srp_bits(0, min(dhi1 - base, kWin - 1));
            if (CLUSTER && a.groups == 2) {   // even or odd offsets
                m0 &= group ? 0xaaaaaaaau : 0x55555555u;
                m1 &= group ? 0xaaaaaaaau : 0x55555555u;
            }
            uint32_t need = __reduce_or_sync(0xffffffffu, m0 | m1);
            const int distinct = __popc(need);
            if (distinct > kSrpShared &&
                distinct > 3 * (int)__reduce_max_sync(0xffffffffu, (unsigned)max(__popc(m0), __popc(m1)))) {
                // scattered estimates (no match, occlusion): each lane takes its own pixels' candidates,
                // from the strip's columns around them
                uint32_t alo[K + 1], ahi[K + 1];
#pragma unroll
                for (int x = 0; x <= RHO; ++x)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        alo[2 * x + c] = __shfl_down_sync(0xffffffffu, ac.lo[c], x);
                        ahi[2 * x + c] = __shfl_down_sync(0xffffffffu, ac.hi[c], x);
                    }
                while (__any_sync(0xffffffffu, (m0 | m1) != 0u)) {
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        uint32_t &m = p ? m1 : m0;
                        const bool on = m != 0u;
                        const int d = base + (on ? __ffs((int)m) - 1 : 0);
                        m &= m - 1u;
                        // a pixel without a candidate left reads the first entries instead
                        const int e = on ? q + p + (dir == 0 ? -d : d) : 0;
                        const uint32_t at = buf + 16u * (uint32_t)(e >> 1);
                        const uint32_t ev = at + ((e & 1) ? odd : 0u), od = at + ((e & 1) ? 16u : odd);
                        const uint4 first = srp_lds(ev);
                        unsigned P0 = __dp4a(alo[p], first.x, 0u), P1 = __dp4a(ahi[p], first.y, 0u);
#pragma unroll
                        for (int k = 1; k < K; ++k) {
                            const uint2 b = srp_lds2((k & 1) ? od + 16u * (uint32_t)(k >> 1) : ev + 16u * (uint32_t)(k >> 1));
                            P0 = __dp4a(alo[p + k], b.x, P0);
                            P1 = __dp4a(ahi[p + k], b.y, P1);
                        }
                        const int N = NB * (int)(P0 + P1) - (p ? sa1 : sa0) * (int)first.z;
                        const float s = on ? __fmul_rn((float)N, __uint_as_float(first.w)) : kNone;
                        if (p == 0)
                            consider(s, d, b0, r0, d0);
                        else
                            consider(s, d, b1, r1, d1);
                    }
                }
                continue;
            }
            while (need) {
                // a few disparities at a time: their chains of loads, dot products and shuffles overlap
                uint32_t low[kBatch];
                int d[kBatch], x0[kBatch], x1[kBatch], P0[kBatch], P1[kBatch];
                uint4 c0[kBatch], c1[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    low[k] = need & (0u - need);   // 0 when the batch is not full: d repeats, no pixel takes it
                    need ^= low[k];
                    d[k] = low[k] ? base + 31 - __clz((int)low[k]) : d[k ? k - 1 : 0];
                    const int e = dir == 0 ? -d[k] : d[k];
                    const uint32_t at = lane_ent + (uint32_t)(16 * (e >> 1));
                    c0[k] = srp_lds(at + ((e & 1) ? odd : 0u));
                    c1[k] = srp_lds(at + ((e & 1) ? 16u : odd));
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    x0[k] = (int)__dp4a(ac.hi[0], c0[k].y, __dp4a(ac.lo[0], c0[k].x, 0u));
                    x1[k] = (int)__dp4a(ac.hi[1], c1[k].y, __dp4a(ac.lo[1], c1[k].x, 0u));
                }
                srp_block_sums<RHO, kBatch>(x0, x1, P0, P1);
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const int N0 = NB * P0[k] - sa0 * (int)c0[k].z, N1 = NB * P1[k] - sa1 * (int)c1[k].z;
                    const float s0 = __fmul_rn((float)N0, __uint_as_float(c0[k].w));
                    const float s1 = __fmul_rn((float)N1, __uint_as_float(c1[k].w));
                    consider((m0 & low[k]) ? s0 : kNone, d[k], b0, r0, d0);
                    consider((m1 & low[k]) ? s1 : kNone, d[k], b1, r1, d1);
                }
            }
        }
        if (CLUSTER && a.groups == 2) {
            float *at = half + strip * 32 + lane;
            const int n = nw * 32;
            if (group) {
                at[0] = b0;
                at[n] = r0;
                at[2 * n] = __int_as_float(d0);
                at[3 * n] = b1;
                at[4 * n] = r1;
                at[5 * n] = __int_as_float(d1);
                asm volatile("bar.arrive %0, 64;" ::"r"(1 + strip) : "memory");
            } else {
                asm volatile("bar.sync %0, 64;" ::"r"(1 + strip) : "memory");
                auto merge = [](float b, float r, int d, float &best, float &second, int &dbest) {
                    second = fmaxf(fmaxf(second, r), fminf(best, b));
                    dbest = b > best || (b == best && d < dbest) ? d : dbest;
                    best = fmaxf(best, b);
                };
                merge(at[0], at[n], __float_as_int(at[2 * n]), b0, r0, d0);
                merge(at[3 * n], at[4 * n], __float_as_int(at[5 * n]), b1, r1, d1);
            }
        }
        if (group == 0) {
        // 2.25 |b| covers |s1| + |s2| of scores this close; equal zeros keep the first
        constexpr float kEps = 2.25f * 9.5367431640625e-07f;   // 2^-20
        const bool close0 = in0 && r0 > __fmaf_rn(fabsf(b0), -kEps, b0);
        const bool close1 = in1 && r1 > __fmaf_rn(fabsf(b1), -kEps, b1);
        // The instance for few pairs and 7 x 7 blocks is at its register limit and slower with the state of the warp's
        // form at hand (one pair of 1242 x 375: 902 us, 952 with it); the others are faster with it (64 pairs: 1619 us,
        // 1705 without; one pair with 5 x 5 blocks: 935 and 1045).
        if constexpr (WARPS == kSrpFewWarps && RHO == 3) {
            if (close0)
                d0 = srp_exact_best<RHO>(a, v, u0, l00, l01, l02, t, dhi0);
            if (close1)
                d1 = srp_exact_best<RHO>(a, v, u0 + 1, l01, l11, l12, t, dhi1);
        } else if (__any_sync(0xffffffffu, close0 || close1)) {
            const int2 d = srp_settle<RHO>(ac.lo[0], ac.lo[1], ac.hi[0], ac.hi[1],
                                           SrpRow{buf, odd, q, dir, t, {sa0, sa1}, {dhi0, dhi1},
                                                  {{l00, l01, l02}, {l01, l11, l12}}, {d0, d1}, {close0, close1}});
            d0 = d.x;
            d1 = d.y;
        }
        if (mine)
            lv[(v & 1) * n_lv + 1 + pair] = (uint32_t)(in0 ? d0 & 0xffff : 0xffff) | ((in1 ? (uint32_t)d1 : 0xffffu) << 16);
        if (st0)
            out[(size_t)v * W + u0] = (int16_t)d0;
        if (st1)
            out[(size_t)v * W + u0 + 1] = (int16_t)d1;
        }
        // A moves up a row
        ac.push(0, an[0][0]);
        ac.push(1, an[0][1]);
        srp_block_sums<RHO, 1>(&ac.s[0], &ac.s[1], &sa0, &sa1);
        an[0][0] = an[1][0];
        an[0][1] = an[1][1];
        load2(pa, acol, v - RHO - 3 >= 0, an[1]);
        pa -= W;
        }
        if constexpr (CLUSTER) {
            const int step = vb - v + 1;                     // rows done
            if (step % kSrpHalo == 0 && v > RHO) {
                const int par = (step / kSrpHalo) & 1;
                const uint32_t box = (uint32_t)__cvta_generic_to_shared(inbox) + (uint32_t)(par * 2 * kSrpHalo * 2);
                auto send = [&](int to, int slot, int val) {
                    uint32_t r;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(box + 2u * (uint32_t)slot), "r"(to));
                    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(r), "h"((short)val) : "memory");
                };
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int u = u0 + c, val = c ? d1 : d0;
                    if (!(c ? st1 : st0))
                        continue;
                    if (rank > 0 && u < own0 + kSrpHalo)                  // the left neighbour's right halo
                        send(rank - 1, kSrpHalo + (u - own0), val);
                    if (rank + 1 < nrank && u >= own1 - kSrpHalo)         // the right neighbour's left halo
                        send(rank + 1, u - (own1 - kSrpHalo), val);
                }
                cluster_sync_all();
                // the received estimates replace the stale ones of the halo (int16 entries of the pair words)
                int16_t *row = reinterpret_cast<int16_t *>(lv + (v & 1) * n_lv + 1);
                const int16_t *in = inbox + par * 2 * kSrpHalo;
                if (tid < kSrpHalo && rank > 0)
                    row[tid] = in[tid];
                if (tid >= kSrpHalo && tid < 2 * kSrpHalo && rank + 1 < nrank && own1 + tid - kSrpHalo <= umax)
                    row[own1 - px0 + tid - kSrpHalo] = in[tid];
            }
        }
        __syncthreads();
    }
}

// Launch shape of k_srp for maps of W columns.
struct SrpShape {
    int ctas, strips, groups, warps, prep;   // CTAs per map; strips, search groups, warps and strips per preparing warp of a CTA
    int per, extra;
    size_t smem;
};
inline SrpShape srp_shape_of(int W, int rho, int dmax, int ctas)
{
    const int S = srp_strip(rho), V = W - 2 * rho, most = kSrpMaxWarps;
    SrpShape s;
    s.ctas = ctas;
    s.per = (V + ctas - 1) / ctas;
    const int span = s.per + (ctas > 1 ? 2 * kSrpHalo : 0);
    s.strips = (span + S - 1) / S;
    s.extra = ((dmax < W ? dmax : W) + S - 1) / S;
    s.groups = 1;
    s.warps = s.strips;
    s.prep = 1;              // one CTA's own strips hold every column of the other image
    if (ctas > 1) {
        const int all = s.strips + s.extra;
        s.groups = 2 * s.strips + (all + 1) / 2 <= most ? 2 : 1;   // named barriers 1 .. strips, at most 12
        const int room = most - s.groups * s.strips;
        const int np = all < room ? all : room;
        s.prep = np > 0 ? (all + np - 1) / np : kSrpPrep + 1;
        s.warps = s.groups * s.strips + (np > 0 ? np : 0);
    }
    const size_t ent = 2 * 16 * (size_t)srp_entries(s.strips, s.extra, rho);
    s.smem = ent + 2 * 4 * (size_t)(s.strips * (S / 2) + 2) + 2 * 4 * kSrpHalo + 6 * 4 * 32 * (size_t)s.strips;
    return s;
}
// One CTA per map fills the GPU from about 76 maps on (38 pairs); one pair takes 1.57 ms that way and 0.89 ms on
// two clusters of 8 (1242 x 375).  So below that number a map is split over the largest
// cluster whose CTAs still find an SM each, every one keeping at least 96 pixels.  Frames wider than a CTA's
// warps hold are always split.
inline bool srp_fits(const SrpShape &s) { return s.warps <= kSrpMaxWarps && s.prep <= kSrpPrep; }
inline SrpShape srp_shape(int W, int rho, int dmax, int n, int sms)
{
    int c = 8;
    while (c > 1 && (2 * n * c > sms || (W - 2 * rho) / c < 96 || !srp_fits(srp_shape_of(W, rho, dmax, c))))
        c /= 2;
    while (c < 8 && !srp_fits(srp_shape_of(W, rho, dmax, c)))
        c *= 2;
    return srp_shape_of(W, rho, dmax, c);
}

// A warp per row, eight loads in flight per lane; the right map's gathers stay within d_max of the row's own
// columns.  Bound by memory latency: 238 MB in 67 us for 64 x 1242x375 (110 us with a 64-bit division per
// pixel to find its column).
__global__ void __launch_bounds__(256) k_lrc(const int16_t *lf, const int16_t *rt, int W, int rows, int tr, float *disp)
{
    const int lane = threadIdx.x & 31;
    const int step = gridDim.x * (blockDim.x >> 5);
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += step) {
        const int16_t *lr = lf + (size_t)r * W, *rr = rt + (size_t)r * W;
        float *dr = disp + (size_t)r * W;
        for (int c = lane; c < W; c += 32 * 8) {
            int l[8], q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                l[k] = c + 32 * k < W ? (int)__ldg(lr + c + 32 * k) : 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int x = c + 32 * k - l[k];
                q[k] = c + 32 * k < W && x >= 0 ? (int)__ldg(rr + x) : 0x4000;   // outside: no agreement
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (c + 32 * k < W)
                    dr[c + 32 * k] = q[k] != 0x4000 && abs(l[k] - q[k]) <= tr ? (float)l[k] : 0.0f;
        }
    }
}

}  // namespace
}  // namespace ld

struct ld_stereo {
    ld_handle *h = nullptr;
    ld_stereo_params sp{};
    int max_w = 0, max_h = 0, max_n = 0;
    void *mem = nullptr;
    int16_t *lf = nullptr, *rt = nullptr;
    float *disp = nullptr;
    int last_w = 0, last_h = 0, last_n = 0;
    bool have_last = false;
    cudaEvent_t ev[3] = {};
    std::string err;
};

namespace {

std::string g_stereo_error;

int sfail(ld_stereo *st, int code, const std::string &msg)
{
    if (st)
        st->err = msg;
    else
        g_stereo_error = msg;
    return code;
}

int scuda(ld_stereo *st, cudaError_t e, const char *what)
{
    return sfail(st, LD_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

int check_pair(ld_stereo *st, const void *left, const void *right, int w, int hh, int n, const void *out)
{
    if (!left || !right || !out)
        return sfail(st, LD_E_ARG, "null buffer");
    if (w < 16 || hh < 16 || w > st->max_w || hh > st->max_h)
        return sfail(st, LD_E_ARG, "frame size outside [16, max_w] x [16, max_h]");
    if (n < 1 || n > st->max_n)
        return sfail(st, LD_E_ARG, "n_frames outside [1, max_batch]");
    return LD_OK;
}

template <int RHO, int NPREP, bool CLUSTER, int WARPS>
cudaError_t launch_srp_t(const ld::SrpArgs &a, const ld::SrpShape &sh, int n, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sh.ctas, n, 2);
    cfg.blockDim = dim3(32 * sh.warps);
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sh.ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CLUSTER ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, ld::k_srp<RHO, NPREP, CLUSTER, WARPS>, a);
}

template <int RHO>
cudaError_t launch_srp(ld::SrpArgs a, int n, cudaStream_t s)
{
    const ld::SrpShape sh = ld::srp_shape(a.W, RHO, a.dmax, n, ld::sm_count());
    a.per = sh.per;
    a.strips = sh.strips;
    a.n_extra = sh.extra;
    a.groups = sh.groups;
    if (sh.ctas == 1)
        return launch_srp_t<RHO, 1, false, ld::kSrpMaxWarps>(a, sh, n, s);
    if (sh.prep <= 1 && sh.warps <= ld::kSrpFewWarps)
        return launch_srp_t<RHO, 1, true, ld::kSrpFewWarps>(a, sh, n, s);
    return sh.prep <= 2 ? launch_srp_t<RHO, 2, true, ld::kSrpMaxWarps>(a, sh, n, s)
                        : launch_srp_t<RHO, ld::kSrpPrep, true, ld::kSrpMaxWarps>(a, sh, n, s);
}

// The instances launch_srp can choose, allowed all of the device's shared memory once: they are shared by every handle
// of the device, so an allowance that followed each call's own need could fall below another thread's launch.
template <int RHO>
cudaError_t setup_srp(int smem_optin)
{
    cudaError_t e = ld::allow_max_smem(ld::k_srp<RHO, 1, false, ld::kSrpMaxWarps>, smem_optin);
    if (e == cudaSuccess)
        e = ld::allow_max_smem(ld::k_srp<RHO, 1, true, ld::kSrpFewWarps>, smem_optin);
    if (e == cudaSuccess)
        e = ld::allow_max_smem(ld::k_srp<RHO, 2, true, ld::kSrpMaxWarps>, smem_optin);
    if (e == cudaSuccess)
        e = ld::allow_max_smem(ld::k_srp<RHO, ld::kSrpPrep, true, ld::kSrpMaxWarps>, smem_optin);
    return e;
}

// both maps and the check on the handle's stream; `timed` records an event before SRP, between, after LRC
int enqueue_stereo(ld_stereo *st, const uint8_t *left, const uint8_t *right, int w, int hh, int n, float *disp,
                   bool timed)
{
    cudaStream_t s = ld::handle_stream(st->h);
    cudaError_t e = cudaSuccess;
    if (timed && (e = cudaEventRecord(st->ev[0], s)) != cudaSuccess)
        return scuda(st, e, "event");
    ld::SrpArgs a{left, right, st->lf, st->rt, w, hh, st->sp.d_max, st->sp.tau, 0, 0, 0, 0};
    switch (st->sp.rho) {
    case 1: e = launch_srp<1>(a, n, s); break;
    case 2: e = launch_srp<2>(a, n, s); break;
    default: e = launch_srp<3>(a, n, s); break;
    }
    if (e != cudaSuccess)
        return scuda(st, e, "search range propagation");
    if (timed && (e = cudaEventRecord(st->ev[1], s)) != cudaSuccess)
        return scuda(st, e, "event");
    const int rows = n * hh, g = (rows + 7) / 8, gmax = ld::sm_count() * 8;
    ld::k_lrc<<<g < gmax ? g : gmax, 256, 0, s>>>(st->lf, st->rt, w, rows, st->sp.tr_lrc, disp);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return scuda(st, e, "consistency check");
    if (timed && (e = cudaEventRecord(st->ev[2], s)) != cudaSuccess)
        return scuda(st, e, "event");
    st->last_w = w;
    st->last_h = hh;
    st->last_n = n;
    st->have_last = true;
    return LD_OK;
}

}  // namespace

extern "C" {

void ld_stereo_params_default(ld_stereo_params *sp)
{
    if (!sp)
        return;
    std::memset(sp, 0, sizeof(*sp));
    sp->rho = 3;
    sp->tau = 1;
    sp->d_max = -1;
    sp->tr_lrc = 3;
}

int ld_stereo_create(ld_handle *h, const ld_stereo_params *sp, ld_stereo **out)
{
    if (!out)
        return sfail(nullptr, LD_E_ARG, "out is NULL");
    *out = nullptr;
    if (!h || !sp)
        return sfail(nullptr, LD_E_ARG, "null argument");
    if (sp->rho < 1 || sp->rho > 3 || sp->tau < 0 || sp->tau > 64 || sp->tr_lrc < 0 || sp->d_max < -1 ||
        sp->d_max > 1023)
        return sfail(nullptr, LD_E_ARG, "rho must be in [1, 3], tau in [0, 64], tr_lrc >= 0, d_max in [-1, 1023]");
    ld_stereo *st = new ld_stereo();
    st->h = h;
    st->sp = *sp;
    if (st->sp.d_max < 0)
        st->sp.d_max = ld::handle_params(h).n_disp - 1;
    ld::handle_dims(h, &st->max_w, &st->max_h, &st->max_n);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = sp->rho == 1 ? setup_srp<1>(optin) : sp->rho == 2 ? setup_srp<2>(optin) : setup_srp<3>(optin);
    if (e != cudaSuccess) {
        delete st;
        return scuda(nullptr, e, "kernel set-up");
    }
    const size_t px = (size_t)st->max_n * st->max_w * st->max_h;
    if (e == cudaSuccess)
        e = cudaMalloc(&st->mem, px * (2 + 2 + 4) + 512);
    if (e != cudaSuccess) {
        cudaGetLastError();
        delete st;
        return sfail(nullptr, LD_E_NOMEM, std::string("stereo memory: ") + cudaGetErrorString(e));
    }
    char *b = (char *)st->mem;
    st->lf = (int16_t *)b;
    st->rt = (int16_t *)(b + ((px * 2 + 255) & ~(size_t)255));
    st->disp = (float *)(b + 2 * ((px * 2 + 255) & ~(size_t)255));
    for (int k = 0; k < 3 && e == cudaSuccess; ++k)
        e = cudaEventCreate(&st->ev[k]);
    if (e != cudaSuccess) {
        scuda(nullptr, e, "event creation");
        ld_stereo_destroy(st);
        return LD_E_CUDA;
    }
    *out = st;
    return LD_OK;
}

int ld_stereo_run(ld_stereo *st, const uint8_t *left, const uint8_t *right, int32_t w, int32_t hh, int32_t n,
                  float *disp_out)
{
    if (!st)
        return LD_E_ARG;
    int rc = check_pair(st, left, right, w, hh, n, disp_out);
    return rc != LD_OK ? rc : enqueue_stereo(st, left, right, w, hh, n, disp_out, false);
}

int ld_stereo_run_timed(ld_stereo *st, const uint8_t *left, const uint8_t *right, int32_t w, int32_t hh, int32_t n,
                        float *disp_out, float *ms_out)
{
    if (!st)
        return LD_E_ARG;
    int rc = check_pair(st, left, right, w, hh, n, disp_out);
    if (rc == LD_OK && !ms_out)
        rc = sfail(st, LD_E_ARG, "ms_out is NULL");
    if (rc == LD_OK)
        rc = enqueue_stereo(st, left, right, w, hh, n, disp_out, true);
    if (rc != LD_OK)
        return rc;
    cudaError_t e = cudaEventSynchronize(st->ev[2]);
    if (e == cudaSuccess)
        e = cudaEventElapsedTime(&ms_out[0], st->ev[0], st->ev[1]);
    if (e == cudaSuccess)
        e = cudaEventElapsedTime(&ms_out[1], st->ev[1], st->ev[2]);
    return e == cudaSuccess ? LD_OK : scuda(st, e, "event timing");
}

int ld_detect_stereo(ld_stereo *st, const uint8_t *left, const uint8_t *right, int32_t w, int32_t hh, int32_t n,
                     ld_lanes *out_lanes)
{
    if (!st)
        return LD_E_ARG;
    int rc = check_pair(st, left, right, w, hh, n, out_lanes);
    if (rc == LD_OK)
        rc = enqueue_stereo(st, left, right, w, hh, n, st->disp, false);
    if (rc != LD_OK)
        return rc;
    rc = ld_detect(st->h, st->disp, left, w, hh, n, out_lanes);
    return rc == LD_OK ? LD_OK : sfail(st, rc, ld_last_error(st->h));
}

int ld_stereo_maps(ld_stereo *st, int32_t frame, int16_t *lf_host, int16_t *rt_host, float *disp_host)
{
    if (!st)
        return LD_E_ARG;
    if (!st->have_last)
        return sfail(st, LD_E_STATE, "no stereo call yet");
    if (frame < 0 || frame >= st->last_n)
        return sfail(st, LD_E_ARG, "frame out of range");
    cudaError_t e = cudaStreamSynchronize(ld::handle_stream(st->h));
    const size_t px = (size_t)st->last_w * st->last_h, o = (size_t)frame * px;
    if (e == cudaSuccess && lf_host)
        e = cudaMemcpy(lf_host, st->lf + o, px * 2, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && rt_host)
        e = cudaMemcpy(rt_host, st->rt + o, px * 2, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && disp_host)
        e = cudaMemcpy(disp_host, st->disp + o, px * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? LD_OK : scuda(st, e, "map copy");
}

const char *ld_stereo_last_error(const ld_stereo *st) { return st ? st->err.c_str() : g_stereo_error.c_str(); }

void ld_stereo_destroy(ld_stereo *st)
{
    if (!st)
        return;
    cudaStreamSynchronize(ld::handle_stream(st->h));
    for (int k = 0; k < 3; ++k)
        if (st->ev[k])
            cudaEventDestroy(st->ev[k]);
    cudaFree(st->mem);
    delete st;
}

}  // extern "C"
