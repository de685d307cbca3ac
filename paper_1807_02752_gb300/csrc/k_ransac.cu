// RANSAC least-squares fits, one CTA per frame:
//
//   k_fit<3>  Alg. 4 on the road DP path M_y (points (v_d, d)), least squares fit of Eq. 13 -> beta; then
//             the first road row f^-1(0) on the row grid and, per road row, f(v) and V_py(v) (Eq. 14).
//   k_fit<5>  Alg. 6 on the V_px DP path M_x (points (v, u_v)), fit of Eq. 19 / Eq. 20 -> gamma; then
//             V_px(v) (Eq. 22) per road row.
//
// Reading of the loop of Alg. 4 / Alg. 6 (draw a random sample, fit it, count inliers, drop the outliers,
// repeat until the inlier fraction reaches eps, then fit the inliers):
//   - each round draws `hyps` minimal samples (M points) from the working set S, listed in increasing point
//     index; draw j takes word j & 3 of Philox4x32-10 at counter (stage << 24 | round, hypothesis, j >> 2, 0)
//     with key = seed, and picks list position floor(word * |S| / 2^32); a draw repeating a chosen point or a
//     chosen row is skipped, and after 8 M draws without M points the hypothesis is void;
//   - the sample is fitted exactly (for M points the least squares fit is the interpolant): Newton divided
//     differences in float32 over tau = (v - centre) / 2^e, in draw order;
//   - inliers are points of S with (y - g(v))^2 < tr, g evaluated in float32 in nested Newton form;
//   - the hypothesis with most inliers (lowest index on ties) wins the round and its outliers leave S;
//   - the loop ends after the first round with eps_den n_I >= eps_num |S|, when no hypothesis is valid, or
//     at the round cap; the final fit is least squares over S, by the normal equations of Eq. 20 (exact
//     integer sums over t = v - centre, rounded once to double, scaled by exact powers of two - the kappa of
//     Eq. 20 - and solved in float64 by Gaussian elimination with partial pivoting; a pivot below 2^-40 is
//     singular).
//
// GB300 mapping (one CTA per frame; the stages are chains of latencies):
//   - the working set stays compacted in shared memory in point order, as (x, y) pairs for the draws and the
//     exact sums and as (tau, -y) floats for the inlier test, so a draw is one load and a test one more;
//   - every THREAD fits one hypothesis in float32 (GB300's FP64 pipe is narrow, so float64 is kept to the final
//     solve), the four draws of a Philox block loaded together.  The threads of a hypothesis (four with 64
//     hypotheses) fit it redundantly, which costs less than handing the coefficients over, and share the
//     points of its inlier count, two points per packed float instruction;
//   - every warp finds the round's winner for itself (one max-reduction of count and index), and the working
//     set is compacted with ballots: three barriers a round;
//   - the final sums are formed in 64-bit integers (powers from t^6 on as two halves), reduced over a warp in
//     27-bit limbs by integer reductions; the normal equations are solved on one warp, one column per lane,
//     with one division per elimination step (each lane one factor).
// Measured (GB300), against serial draws with dependent loads, int128 sums and shuffles: k_fit<5> 78 -> 47 us
// and k_fit<3> 27 -> 18 us on 64 x 1242x375, 45 -> 31 and 22 -> 16 us on one such frame.  A round of 64
// hypotheses over 250 points is about 6000 cycles (fitting 2200, counting 2700, the rest barriers and
// compaction); the float64 solve of the quartic is 12 500 cycles (a double addition takes 63 cycles here, a
// division 560) and bounds what is left.
#include "ld_internal.cuh"

namespace ld {

namespace {

constexpr int kFitThreads = 256;
constexpr int kNW = kFitThreads / 32;

__device__ __forceinline__ double p2d(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }

__device__ __forceinline__ long long magnitude(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffll; }

// Normal equations of M unknowns from exact sums S = (Sx[0 .. 2M-2], Sy[0 .. M-1]), Sx[k] = sum t^k,
// Sy[k] = sum y t^k: A[r][c] = Sx[r + c] 2^-(r+c)e, b[r] = Sy[r] 2^-re (exact power-of-two column scaling),
// Gaussian elimination with partial pivoting (first row of largest |pivot|; a pivot below 2^-40 is
// singular), then back substitution; every product, difference and quotient rounded once, no FMA.  Solved
// on one warp: lane j <= M holds column j of the augmented matrix, the pivot column is broadcast with
// shuffles and every lane applies the elimination to its own column (the same operations, in the same
// order, as the serial algorithm); lane 0 back-substitutes.  All lanes of the warp must call it.  Returns
// 0 on every lane, or -1 if singular.
template <int M>
__device__ int solve_normal_warp(const __int128 *S, int e, double *coef)
{
    const int lane = threadIdx.x & 31;
    const int c = lane <= M ? lane : M;  // lanes past M shadow column M and are never read
    double col[M];
#pragma unroll
    for (int r = 0; r < M; ++r)
        col[r] = c < M ? __dmul_rn(i128_to_f64(S[r + c]), p2d(-(r + c) * e))
                       : __dmul_rn(i128_to_f64(S[2 * M - 1 + r]), p2d(-r * e));
#pragma unroll
    for (int k = 0; k < M; ++k) {
        double pc[M];  // column k (after the previous steps), from lane k
#pragma unroll
        for (int i = 0; i < M; ++i)
            pc[i] = __shfl_sync(0xffffffffu, col[i], k);
        // magnitudes compared as integers (finite values order like their bits; a double comparison takes as
        // long as a double addition, 63 cycles)
        int piv = k;
        long long pa = magnitude(pc[k]);
#pragma unroll
        for (int i = k + 1; i < M; ++i)
            if (magnitude(pc[i]) > pa) {
                pa = magnitude(pc[i]);
                piv = i;
            }
        if (pa < magnitude(0x1p-40))
            return -1;
#pragma unroll
        for (int i = k + 1; i < M; ++i)
            if (i == piv) {
                double t = col[k];
                col[k] = col[i];
                col[i] = t;
                t = pc[k];
                pc[k] = pc[i];
                pc[i] = t;
            }
        if (k + 1 < M) {
            // lane i divides for row i; the factors are then handed round
            double num = pc[M - 1];
#pragma unroll
            for (int i = k + 1; i < M - 1; ++i)
                num = lane == i ? pc[i] : num;
            const double fct = __ddiv_rn(num, pc[k]);
#pragma unroll
            for (int i = k + 1; i < M; ++i) {
                const double fi = __shfl_sync(0xffffffffu, fct, i);
                if (c > k)
                    col[i] = __dsub_rn(col[i], __dmul_rn(fi, col[k]));
            }
        }
    }
    // back substitution on lane 0, rows gathered from the column lanes
    double A[M][M + 1];
#pragma unroll
    for (int r = 0; r < M; ++r)
#pragma unroll
        for (int j = 0; j <= M; ++j)
            A[r][j] = __shfl_sync(0xffffffffu, col[r], j);
#pragma unroll
    for (int k = M - 1; k >= 0; --k) {
        double s = A[k][M];
#pragma unroll
        for (int j = k + 1; j < M; ++j)
            s = __dsub_rn(s, __dmul_rn(A[k][j], coef[j]));
        coef[k] = __ddiv_rn(s, A[k][k]);
    }
    return 0;
}

// Sum over the warp of a signed 64-bit integer (whose true sum fits 64 bits), on every lane.
__device__ __forceinline__ long long warp_sum64(long long v)
{
    constexpr unsigned kAll = 0xffffffffu, kLimb = (1u << 27) - 1u;   // 32 limbs of 27 bits fit 32 bits
    const unsigned l0 = __reduce_add_sync(kAll, (unsigned)v & kLimb);
    const unsigned l1 = __reduce_add_sync(kAll, (unsigned)(v >> 27) & kLimb);
    const int l2 = __reduce_add_sync(kAll, (int)(v >> 54));
    return (long long)((unsigned long long)l0 + ((unsigned long long)l1 << 27) + ((unsigned long long)(long long)l2 << 54));
}

template <typename T>
__device__ __forceinline__ T *carve(unsigned char *&p, size_t count)
{
    const size_t off = ((size_t)p + 15) & ~(size_t)15;
    T *r = reinterpret_cast<T *>(off);
    p = reinterpret_cast<unsigned char *>(off + sizeof(T) * count);
    return r;
}

// One hypothesis: the minimal sample of Philox draws from the ns points xy (x << 16 | y) and the polynomial
// through it in Newton form (nodes = the sample's tau in draw order, c = float32 divided differences).
template <int M>
__device__ __forceinline__ bool hypothesis(const KParams &kp, const uint32_t *xy, const float *rcp, int ns, int stage, int round,
                                           int h, float sc, float *c, float *nodes)
{
    int X[M], Y[M];
#pragma unroll
    for (int k = 0; k < M; ++k)
        X[k] = -1, Y[k] = 0;   // no point has x = -1
    int got = 0;
#pragma unroll 1
    for (int b = 0; b < 2 * M && got < M; ++b) {
        const uint4 w = philox4x32_10(make_uint4(((uint32_t)stage << 24) | (uint32_t)round, (uint32_t)h, (uint32_t)b, 0u),
                                      kp.key0, kp.key1);
        const uint32_t wv[4] = {w.x, w.y, w.z, w.w};
        uint32_t p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int idx = (int)__umulhi(wv[q], (uint32_t)ns);
            p[q] = LD_IN(idx, ns, CK_FIT_SAMPLE) ? xy[idx] : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int x = (int)(p[q] >> 16);
            bool take = got < M;   // a point or a row drawn before is skipped
#pragma unroll
            for (int k = 0; k < M; ++k)
                take = take && X[k] != x;
#pragma unroll
            for (int k = 0; k < M; ++k)
                if (take && k == got) {
                    X[k] = x;
                    Y[k] = (int)(p[q] & 0xffffu);
                }
            got += take ? 1 : 0;
        }
    }
    if (got < M)
        return false;
#pragma unroll
    for (int q = 0; q < M; ++q) {
        nodes[q] = __fmul_rn((float)(X[q] - kp.centre), sc);
        c[q] = (float)Y[q];
    }
    // Divided differences.  A divisor is (x_i - x_j) 2^-e, whose reciprocal the table holds correctly rounded,
    // so the quotient takes a product and two remainder corrections (P. Markstein, IBM J. Res. Dev. 34, 1990:
    // from a faithful quotient and the correctly rounded reciprocal, the corrected quotient is the correctly
    // rounded one), without the branch of the general division.  Its remainders are exact unless the dividend
    // is tiny: then the sample is divided in the general way.
    float d[M];
    bool tiny = false;
#pragma unroll
    for (int i = 0; i < M; ++i)
        d[i] = c[i];
#pragma unroll
    for (int k = 1; k < M; ++k)
#pragma unroll
        for (int i = M - 1; i >= k; --i) {
            const int dx = X[i] - X[i - k];
            const float r = rcp[abs(dx)], y = dx < 0 ? -r : r;
            const float num = __fsub_rn(d[i], d[i - 1]), den = __fsub_rn(nodes[i], nodes[i - k]);
            tiny = tiny || (num != 0.0f && fabsf(num) < 0x1p-60f);
            float q = __fmul_rn(num, y);
            q = __fmaf_rn(__fmaf_rn(-q, den, num), y, q);
            d[i] = __fmaf_rn(__fmaf_rn(-q, den, num), y, q);
        }
    if (tiny) {
#pragma unroll
        for (int k = 1; k < M; ++k)
#pragma unroll
            for (int i = M - 1; i >= k; --i)
                c[i] = __fdiv_rn(__fsub_rn(c[i], c[i - 1]), __fsub_rn(nodes[i], nodes[i - k]));
    } else {
#pragma unroll
        for (int i = 0; i < M; ++i)
            c[i] = d[i];
    }
    return true;
}

// Inlier test of a Newton-form hypothesis: (y - p(tau))^2 < tr, nested evaluation in float32 (one rounding per
// operation), for ty = (tau, -y); nn: the negated nodes.
template <int M>
__device__ __forceinline__ bool newton_inlier(const float *c, const float *nn, float2 ty, float tr)
{
    float p = c[M - 1];
#pragma unroll
    for (int k = M - 2; k >= 0; --k)
        p = __fadd_rn(__fmul_rn(p, __fadd_rn(ty.x, nn[k])), c[k]);
    const float r = __fadd_rn(p, ty.y);   // p - y: its square is that of y - p
    return __fmul_rn(r, r) < tr;
}
// Packed product, each half rounded once: a fused multiply-add of minus zero, computed so that the compiler does
// not know its value (a packed multiplication is contracted with a packed addition that follows it, whatever
// the contraction flags say, and a known zero turns the multiply-add back into that multiplication).
__device__ __forceinline__ float2 mul2(float2 a, float2 b, float2 minus_zero) { return __ffma2_rn(a, b, minus_zero); }

// The inlier test of two points at once (packed float: each half rounded as the scalar operation).
template <int M>
__device__ __forceinline__ int newton_inlier2(const float *c, const float *nn, float2 a, float2 b, float tr, float2 mz)
{
    const float2 tau = make_float2(a.x, b.x);
    float2 p = make_float2(c[M - 1], c[M - 1]);
#pragma unroll
    for (int k = M - 2; k >= 0; --k)
        p = __fadd2_rn(mul2(p, __fadd2_rn(tau, make_float2(nn[k], nn[k])), mz), make_float2(c[k], c[k]));
    const float2 r = __fadd2_rn(p, make_float2(a.y, b.y));
    const float2 s = mul2(r, r, mz);
    return (s.x < tr ? 1 : 0) + (s.y < tr ? 1 : 0);
}

template <int M>
__device__ __forceinline__ void fit_body(const KParams &kp, const Work &w, const int f)
{
    constexpr int stage = M == 3 ? 0 : 1;
    constexpr int kPer = (LD_MAX_H + kFitThreads - 1) / kFitThreads;   // points a thread compacts (D <= LD_MAX_H)
    constexpr int NS = 3 * M - 1;   // exact sums: t^k, k <= 2M - 2, then y t^k, k < M
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double coef_s[M];
    __shared__ int sh[4];
    const int H = kp.H, P = w.pmax;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const FrameState fs0 = w.fs[f];
    const int n0 = w.npts[f * 2 + stage];
    const int16_t *gp = w.pts + ((size_t)f * 2 + stage) * 3 * P;

    unsigned char *p = smem;
    uint32_t *xy = carve<uint32_t>(p, P);
    float2 *ty = carve<float2>(p, P);
    int16_t *pid = carve<int16_t>(p, P);
    int *chunk = carve<int>(p, kPer * kNW);
    int *count = carve<int>(p, kMaxHyps);               // inliers of each hypothesis; negative: void
    float *rcp = carve<float>(p, H);                    // 2^e / i, correctly rounded
    float *hyp_cf = carve<float>(p, kMaxHyps * 2 * M);  // per hypothesis: M divided differences, M negated nodes
    __int128 *red = carve<__int128>(p, NS);
    long long *red64 = carve<long long>(p, kNW * (NS + 3));
    int *redc = carve<int>(p, kNW);

    const int centre = kp.centre;
    const float sc = pow2f(-kp.e);
    const float tr = stage == 0 ? kp.tr_y : kp.tr_x;
    for (int i = tid; i < H; i += kFitThreads)
        rcp[i] = __fmul_rn(__frcp_rn((float)max(i, 1)), pow2f(kp.e));
    for (int i = tid; i < kp.hyps; i += kFitThreads)
        count[i] = 0;
    const int most = min(P, stage == 0 ? kp.D : H);         // points there can be (the list's memory holds P)
#pragma unroll 2
    for (int j = tid; j < most; j += kFitThreads) {
        const int x = gp[j], y = gp[P + j];
        xy[j] = (uint32_t)(x & 0xffff) << 16 | (uint32_t)(y & 0xffff);
        ty[j] = make_float2(__fmul_rn((float)(x - centre), sc), -(float)y);
        pid[j] = gp[2 * P + j];
    }
    if (stage == 1 && (fs0.flags & LD_F_NO_LANES))
        return;   // k_vpx_dp wrote no points
    const int n = LD_IN(n0, P + 1, CK_FIT_NPTS) ? n0 : 0;
    const int n_inl = stage == 0 ? kp.D : H;
    uint8_t *inl = stage == 0 ? w.inl_y + (size_t)f * n_inl : w.inl_x + (size_t)f * n_inl;
    for (int i = tid; i < n_inl; i += kFitThreads)
        inl[i] = 0;
    __syncthreads();

    // hypothesis h is fitted and counted by `groups` threads, h + g nh
    const int nh = kp.hyps, groups = min(kFitThreads / nh, 32), h = tid % nh, g = tid / nh;
    const float2 mz = make_float2(__fmul_rn(sc, -0.0f), __fmul_rn(sc, -0.0f));   // -0 (see mul2)
    int fl = 0, round = 0, ns = n;
    for (;;) {
        if (ns < M) {
            fl |= 2;
            break;
        }
        if (round == kp.rounds) {
            fl |= 1;
            break;
        }
        if (g < groups) {
            float c[M], nn[M];
            const bool ok = hypothesis<M>(kp, xy, rcp, ns, stage, round, h, sc, c, nn);
            int cnt = -1;
            if (ok) {
                cnt = 0;
#pragma unroll
                for (int k = 0; k < M; ++k)
                    nn[k] = -nn[k];
                int q = g;
#pragma unroll 4
                for (; q + groups < ns; q += 2 * groups)
                    cnt += newton_inlier2<M>(c, nn, ty[q], ty[q + groups], tr, mz);
                if (q < ns)
                    cnt += newton_inlier<M>(c, nn, ty[q], tr) ? 1 : 0;
                if (g == 0)
#pragma unroll
                    for (int k = 0; k < M; ++k) {
                        hyp_cf[h * 2 * M + k] = c[k];
                        hyp_cf[h * 2 * M + M + k] = nn[k];
                    }
            }
            if (cnt > 0 || (cnt < 0 && g == 0))
                atomicAdd(&count[h], cnt > 0 ? cnt : -(1 << 20));
        }
        __syncthreads();
        // the winner: most inliers, then the lowest index (count << 8 | 255 - index; negative when none is valid)
        int best = -1;
        for (int i = lane; i < nh; i += 32)
            best = max(best, count[i] * 256 + (255 - i));
        best = __reduce_max_sync(0xffffffffu, best);
        ++round;
        if (best < 0) {
            fl |= 2;
            break;
        }
        const int bh = 255 - (best & 255), bc = best >> 8;
        float cf[2 * M];
#pragma unroll
        for (int k = 0; k < 2 * M; ++k)
            cf[k] = hyp_cf[bh * 2 * M + k];
        // the winner's inliers stay, in order: each warp flags its chunks of 32 points, then places them
        uint32_t kxy[kPer];
        float2 kty[kPer];
        int16_t kid[kPer];
        unsigned keep[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int j = tid + i * kFitThreads;
            keep[i] = 0u;
            if (i * kFitThreads >= ns)
                break;
            if (j < ns) {
                kxy[i] = xy[j];
                kty[i] = ty[j];
                kid[i] = pid[j];
            }
            keep[i] = __ballot_sync(0xffffffffu, j < ns && newton_inlier<M>(cf, cf + M, kty[i], tr));
            if (lane == 0)
                chunk[i * kNW + warp] = __popc(keep[i]);
        }
        __syncthreads();
        for (int i = tid; i < nh; i += kFitThreads)
            count[i] = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            if (i * kFitThreads >= ns)
                break;
            const int me = i * kNW + warp;   // chunks before this one
            int before = lane < me ? chunk[lane] : 0;
            if (kPer * kNW > 32 && lane + 32 < me)
                before += chunk[lane + 32];
            before = __reduce_add_sync(0xffffffffu, before);
            if (keep[i] >> lane & 1u) {
                const int at = before + __popc(keep[i] & ((1u << lane) - 1u));
                xy[at] = kxy[i];
                ty[at] = kty[i];
                pid[at] = kid[i];
            }
        }
        const bool done = (long long)kp.eps_den * bc >= (long long)kp.eps_num * ns;
        ns = bc;
        __syncthreads();
        if (done)
            break;
    }
    for (int j = tid; j < ns; j += kFitThreads)   // final membership (cleared before the rounds)
        if (LD_IN(pid[j], n_inl, CK_FIT_ROW))
            inl[pid[j]] = 1;
    // final least squares over the remaining set: exact sums (sum t^k for k <= 2M-2, then sum y t^k for k < M),
    // then the normal equations solved on one warp.  |t| <= LD_MAX_H / 2, y < LD_MAX_W and at most LD_MAX_H points: sums
    // of t^k up to k = 5 and of y t^k up to k = 4 fit 64 bits; t^6 .. t^8 are summed as 2^32 hi + lo.
    constexpr double kT = LD_MAX_H / 2, kT4 = kT * kT * kT * kT;
    static_assert(LD_MAX_D <= LD_MAX_H && LD_MAX_H * LD_MAX_W * kT4 < 9.2e18 && LD_MAX_H * kT4 * kT < 9.2e18 &&
                      LD_MAX_H * kT4 * kT4 / 4294967296.0 < 9.2e18, "exact sums");
    if (!(fl & 2)) {
        constexpr int N64 = 2 * M - 1 > 6 ? 6 : 2 * M - 1;   // powers 0 .. N64 - 1 in 64 bits
        constexpr int NHI = 2 * M - 1 - N64;
        long long sx[N64], sy[M], hi[NHI > 0 ? NHI : 1], lo[NHI > 0 ? NHI : 1];
#pragma unroll
        for (int k = 0; k < N64; ++k)
            sx[k] = 0;
#pragma unroll
        for (int k = 0; k < M; ++k)
            sy[k] = 0;
#pragma unroll
        for (int k = 0; k < NHI; ++k)
            hi[k] = lo[k] = 0;
        for (int j = tid; j < ns; j += kFitThreads) {
            const uint32_t v = xy[j];
            const long long t = (int)(v >> 16) - centre, y = (int)(v & 0xffffu);
            long long pw = 1;
#pragma unroll
            for (int k = 0; k < N64; ++k) {
                sx[k] += pw;
                if (k < M)
                    sy[k] += y * pw;
                if (k + 1 < N64)
                    pw *= t;
            }
            long long q = t;   // t^5 t^(k+1)
#pragma unroll
            for (int k = 0; k < NHI; ++k) {
                const unsigned long long l = (unsigned long long)pw * (unsigned long long)q;
                const long long hh = __mul64hi(pw, q);
                hi[k] += (long long)((unsigned long long)hh << 32 | l >> 32);
                lo[k] += (long long)(l & 0xffffffffull);
                q *= t;
            }
        }
#pragma unroll
        for (int k = 0; k < N64; ++k)
            sx[k] = warp_sum64(sx[k]);
#pragma unroll
        for (int k = 0; k < M; ++k)
            sy[k] = warp_sum64(sy[k]);
#pragma unroll
        for (int k = 0; k < NHI; ++k) {
            hi[k] = warp_sum64(hi[k]);
            lo[k] = warp_sum64(lo[k]);
        }
        if (lane == 0) {
            long long *r = red64 + warp * (NS + 3);
#pragma unroll
            for (int k = 0; k < N64; ++k)
                r[k] = sx[k];
#pragma unroll
            for (int k = 0; k < NHI; ++k) {
                r[N64 + k] = hi[k];
                r[NS + k] = lo[k];
            }
#pragma unroll
            for (int k = 0; k < M; ++k)
                r[2 * M - 1 + k] = sy[k];
        }
        __syncthreads();
        if (warp == 0) {
            if (lane < NS) {
                long long a = 0, b = 0;
                const bool two = lane >= N64 && lane < 2 * M - 1;
                for (int wv = 0; wv < kNW; ++wv) {
                    a += red64[wv * (NS + 3) + lane];
                    if (two)
                        b += red64[wv * (NS + 3) + NS + lane - N64];
                }
                red[lane] = two ? ((__int128)a << 32) + b : (__int128)a;
            }
            __syncwarp();
            double cd[M];
            int ok = ns >= M ? solve_normal_warp<M>(red, kp.e, cd) == 0 : 0;
            if (lane == 0) {
                if (ok)
                    for (int k = 0; k < M; ++k)
                        coef_s[k] = cd[k];
                sh[2] = ok;
            }
        }
        __syncthreads();
        if (!sh[2])
            fl |= 2;
    }

    const double sc64 = p2d(-kp.e);
    if (stage == 0) {
        int flags = 0;
        if (fl & 1)
            flags |= LD_F_CAP_Y;
        if (fl & 2)
            flags |= LD_F_DEGEN_Y;
        double beta[3] = {0.0, 0.0, 0.0};
        int vtop = H;
        float *rows = w.rows + (size_t)f * 3 * H;
        if (!(fl & 2)) {
            for (int i = 0; i < 3; ++i)
                beta[i] = coef_s[i];
            // v_top: first row of the bottom run of rows with f(v) > 0 and f'(v) > 0
            double fv[kPer], dfv[kPer];
            int worst = -1;
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int v = tid + i * kFitThreads;
                if (v >= H)
                    break;
                const double tau = __dmul_rn((double)(v - centre), sc64);
                fv[i] = poly_f64<3>(beta, tau);
                dfv[i] = __dmul_rn(__dadd_rn(beta[1], __dmul_rn(__dmul_rn(2.0, beta[2]), tau)), sc64);
                if (!(fv[i] > 0.0 && dfv[i] > 0.0))
                    worst = max(worst, v);
            }
            worst = __reduce_max_sync(0xffffffffu, worst);
            if (lane == 0)
                redc[warp] = worst;
            __syncthreads();
            if (tid == 0) {
                int m = -1;
                for (int i = 0; i < kNW; ++i)
                    m = max(m, redc[i]);
                sh[3] = m + 1;
            }
            __syncthreads();
            vtop = sh[3];
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int v = tid + i * kFitThreads;
                if (v >= H)
                    break;
                float F = 0.0f, Vy = 0.0f;
                if (v >= vtop) {
                    F = __double2float_rn(fv[i]);
                    Vy = __double2float_rn(__dsub_rn((double)v, __ddiv_rn(fv[i], dfv[i])));
                }
                rows[v] = F;
                rows[H + v] = Vy;
                rows[2 * H + v] = 0.0f;
            }
            if (vtop > H - 1)
                flags |= LD_F_NO_ROAD;
        } else {
            for (int v = tid; v < 3 * H; v += kFitThreads)
                rows[v] = 0.0f;
        }
        if (flags & (LD_F_DEGEN_Y | LD_F_NO_ROAD))
            flags |= LD_F_NO_LANES;
        if (tid == 0) {
            FrameState &fs = w.fs[f];
            fs.flags = flags;
            fs.v_top = vtop;
            fs.rounds_y = round;
            fs.rounds_x = 0;
            for (int i = 0; i < 3; ++i)
                fs.beta[i] = beta[i];
            for (int i = 0; i < 5; ++i)
                fs.gamma[i] = 0.0;
        }
    } else {
        int flags = fs0.flags;
        if (fl & 1)
            flags |= LD_F_CAP_X;
        if (fl & 2)
            flags |= LD_F_DEGEN_X | LD_F_NO_LANES;
        double gamma[5] = {0, 0, 0, 0, 0};
        if (!(fl & 2)) {
            for (int i = 0; i < 5; ++i)
                gamma[i] = coef_s[i];
            float *Vpx = w.rows + (size_t)f * 3 * H + 2 * H;
            for (int v = fs0.v_top + tid; v < H; v += kFitThreads)
                Vpx[v] = __double2float_rn(poly_f64<5>(gamma, __dmul_rn((double)(v - centre), sc64)));
        }
        if (tid == 0) {
            FrameState &fs = w.fs[f];
            fs.flags = flags;
            fs.rounds_x = round;
            for (int i = 0; i < 5; ++i)
                fs.gamma[i] = gamma[i];
        }
    }
}

template <int M>
__global__ void __launch_bounds__(kFitThreads) k_fit(const KParams kp, const Work w) { fit_body<M>(kp, w, blockIdx.x); }
template <int M>
__global__ void __launch_bounds__(kFitThreads) k_fit_fd(const FrameDesc *__restrict__ fd)
{
    const FrameDesc &d = fd[blockIdx.x];
    const KParams kp = d.kp;   // the frame's parameters, loaded once into registers
    const Work w = d.w;
    fit_body<M>(kp, w, 0);
}

template <int M>
size_t fit_smem(int P, int H)
{
    size_t s = 0;
    auto add = [&](size_t bytes) { s = ((s + 15) & ~(size_t)15) + bytes; };
    add(4 * (size_t)P);
    add(8 * (size_t)P);
    add(2 * (size_t)P);
    add(4 * ((LD_MAX_H + kFitThreads - 1) / kFitThreads) * kNW);
    add(4 * kMaxHyps);
    add(4 * (size_t)H);
    add(4 * kMaxHyps * 2 * M);
    add(16 * (3 * M - 1));
    add(8 * kNW * (3 * M + 2));
    add(4 * kNW);
    return s + 16;
}

}  // namespace

cudaError_t setup_ransac(int smem_optin)
{
    cudaError_t e = allow_max_smem(k_fit<3>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_fit_fd<3>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_fit_fd<5>, smem_optin);
    if (e == cudaSuccess)
        e = allow_max_smem(k_fit<5>, smem_optin);
    return e;
}

cudaError_t launch_fit_y(const KParams &kp, const Work &w, cudaStream_t s)
{
    k_fit<3><<<kp.n_frames, kFitThreads, fit_smem<3>(w.pmax, kp.H), s>>>(kp, w);
    return cudaGetLastError();
}

cudaError_t launch_fit_y_fd(const KParams &kmax, const FrameDesc *fd, int n, cudaStream_t s)
{
    k_fit_fd<3><<<n, kFitThreads, fit_smem<3>(kmax.pmax_hint, kmax.H), s>>>(fd);
    return cudaGetLastError();
}

cudaError_t launch_fit_x_fd(const KParams &kmax, const FrameDesc *fd, int n, cudaStream_t s)
{
    k_fit_fd<5><<<n, kFitThreads, fit_smem<5>(kmax.pmax_hint, kmax.H), s>>>(fd);
    return cudaGetLastError();
}

cudaError_t launch_fit_x(const KParams &kp, const Work &w, cudaStream_t s)
{
    k_fit<5><<<kp.n_frames, kFitThreads, fit_smem<5>(w.pmax, kp.H), s>>>(kp, w);
    return cudaGetLastError();
}

}  // namespace ld
