/*
 * td_fan.cuh -- the filtered sweep for effective dimensions D = 3 .. 6: the
 * subsets that share all points but one, taken together.
 *
 * Consecutive colex positions S = {c_0 < c_1 < .. < c_(K-1)} (K = D - 2)
 * share the tail (c_1, .., c_(K-1)) while c_0 runs from 0 to c_1 - 1; such a
 * run is called a fan.  Projecting along span(S) can be done in two steps:
 * first along the tail, R^D -> R^3, once for the fan (exact integers), then
 * along the one remaining point.  A team of T warps takes a fan in three
 * stages, each of which leaves fewer subsets to the next:
 *
 *   td_fan_strips  lower bounds of G for all subsets of the fan from tables
 *                  over angular strips of the 3-D quotient: a number of steps
 *                  per point of the fan, not per point and subset;
 *   td_fan_quad    four subsets in one pass over the points: two multiply-
 *                  adds a point and subset, 256 angular rows;
 *   td_sweep_one   one subset with the exact steps.
 *
 * What it is bound by: on the p = 4, n = 1000 data set a subset costs about 52
 * warp instructions in a call of 4 queries (a sweep of the points for two subsets
 * at a time: 779), 96% of the subsets are decided by the strips,
 * issue is active 41% of the time with 16 warps an SM, and the waits are for
 * shared memory (look-ups and histogram updates at random bins) and at the
 * team's barriers; DRAM is idle.  64 queries: 30.1 ms a call before, 3.4 to 3.6
 * now; p = 5, n = 200, 256 queries 138 and 29; p = 6, n = 120, 8 queries 35.9
 * and 12.4; p = 3, n = 1000, 1000 queries 4.37 and 0.80.  On data of a few
 * values, where most subsets go to the exact steps, a team waits for its
 * slowest warp, and calls can be slower than with warps on their own (127
 * queries of p = 3, n = 1403, coordinates -2 .. 2: 13.7 and 33 ms).
 */
#pragma once

/* Rows of a quad's histograms: 256 per subset, plus one word that takes the
 * uncertain points (never read: a store to it costs less than a branch around
 * it).  Bytes per subset, a multiple of 16. */
#define TD_FAN_ROWS 256
#define TD_FAN_TABLE ((TD_FAN_ROWS + 4) * 4)

/* Strip tables (td_fan_strips): words per strip of NB bins, with 4 words of
 * padding before and after: two arrays of 16-bit pairs, or one of 8-bit fours
 * for rows of at most 255 points.  A team's histogram storage, TD_FAN_HIST
 * bytes or more per warp, holds 8 packed strips of 128 bins for one warp, 4
 * unpacked ones of 128 (one warp) or 256 bins (two), 8 of 256 for four. */
#define TD_STRIP_WORDS(bins, packed) ((packed) ? (bins) + 8 : 2 * (bins) + 8)
#define TD_STRIP_MAX 64 /* strips, at most */
#define TD_STRIP_FIRST(D) ((D) == 3 ? 16 : 8) /* to begin with */
#define TD_FAN_HIST (8 * TD_STRIP_WORDS(128, true) * 4)
static_assert(TD_FAN_HIST % 128 == 0 && 4 * TD_STRIP_WORDS(128, false) * 4 <= TD_FAN_HIST &&
                  2 * TD_STRIP_WORDS(256, false) * 4 <= TD_FAN_HIST && 4 * TD_FAN_TABLE <= TD_FAN_HIST,
              "warp histogram storage");

/* Points per warp of a team, times D - 2 (td_fan_team).  48 made the 16-dataset
 * batch 117 ms against 94, 192 made W2 5.4 ms against 3.5. */
#define TD_FAN_SPREAD 96

/* td_fan_strips keeps a flag for each of a warp's blocks of 32 points in a
 * 32-bit word: the longest rows of every team size (td_fan_team), at the widest
 * spread and for the largest teams, have at most 32 blocks a warp. */
static_assert(2 * TD_FAN_SPREAD * (6 - 2) - 1 <= 32 * 32, "flags of a warp's blocks: teams below the largest");
static_assert(TD_MAX_N <= 32 * 32 * td_sweep_warps(3) && TD_MAX_N <= 32 * 32 * td_sweep_warps(4) &&
                  TD_MAX_N <= 32 * 32 * td_sweep_warps(5) && TD_MAX_N <= 32 * 32 * td_sweep_warps(6),
              "flags of a warp's blocks: the largest teams");

__device__ __forceinline__ td_f2x td_fma2_rm(td_f2x a, td_f2x b, td_f2x c)
{
    td_f2x d;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ td_f2x td_lds64(unsigned a)
{
    td_f2x v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a));
    return v;
}

__device__ __forceinline__ uint32_t td_lds32(unsigned a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void td_lds_coef(unsigned a, td_f2x &x, td_f2x &y)
{
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a));
}

/* shared reduction at byte offset OFF from a */
template <int OFF>
__device__ __forceinline__ void td_reds_at(unsigned a, unsigned v)
{
    asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(OFF) : "memory");
}

/* Warps per team for rows of nnz points, a power of two: a team meets at
 * barriers in every stage of a fan, so that warps work alone (T = 1) where a
 * row is short, and the team's planes and tables are shared by more warps
 * where it is long.  At D = 3 the whole tile is one fan. */
__host__ __device__ inline int td_fan_team(int D, int nnz, int warps)
{
    if (D == 3) return warps;
    int t = 1;
    while (2 * t <= warps && 2 * t * TD_FAN_SPREAD * (D - 2) <= nnz) t *= 2;
    return t;
}

/* A team's area: three coordinate planes of the projected points (binary32,
 * zeros up to a multiple of 32) and the list of the fan's c_0 values.
 * Multiples of 128 bytes. */
__host__ __device__ inline int td_fan_plane(int nnz) { return (nnz + 31) & ~31; }

__host__ __device__ inline size_t td_fan_area(int nnz)
{
    const int ny = td_fan_plane(nnz);
    return ((size_t)ny * 12 + (size_t)(ny + 16) * 2 + 127) & ~(size_t)127;
}

/* Bytes of all team areas of a CTA for rows of up to nmax points: a smaller
 * row may be taken by smaller teams, more of them, with smaller areas. */
__host__ __device__ inline size_t td_fan_areas(int D, int nmax, int warps)
{
    size_t most = 0;
    const int tmax = td_fan_team(D, nmax, warps);
    for (int t = 1; t <= tmax; t *= 2) {
        /* the longest row that teams of t warps take */
        int n = nmax;
        if (t < tmax && 2 * t * TD_FAN_SPREAD * (D - 2) - 1 < n) n = 2 * t * TD_FAN_SPREAD * (D - 2) - 1;
        if (D == 3 && t < warps) continue;
        const size_t b = (size_t)(warps / t) * td_fan_area(n);
        if (b > most) most = b;
    }
    return most;
}

/* Per-team state in shared memory. */
struct TdFanHead {
    int64_t kappa;      /* determinant of the tail on its pivot rows */
    int64_t d[3][4];    /* the same with pivot row j replaced by the r-th other row */
    float fk, fd[3][4]; /* both in binary32 (exact in mode 0) */
    int off[8];         /* staged-layout offsets of the pivot rows [0, K-1) and of the other rows [4, 7) */
    int mode;           /* arithmetic of the projection (td_fan_project); -1: dependent tail */
    int stop;           /* early exit: some warp has reached 0 */
    int next;           /* the team's next fan in the tile */
    unsigned mx;        /* bit pattern of the largest |Y| */
};

/* A warp's contribution to its team's fan, in its basis block. */
struct TdFanPart {
    int left, dependent; /* c_0 values to sweep one by one, and dependent ones */
    float sum[3]; /* sums of |Y| by coordinate */
};
static_assert(16 + TD_WARP_BASIS_BYTES + 9 * 8 + sizeof(TdFanPart) <= TD_WARP_BLOCK_BYTES, "warp block");

/* A team, as byte offsets into the dynamic shared memory (32-bit, and known
 * to be shared to the compiler, where pointers kept across the fan loop would
 * take twice the registers). */
struct TdFan {
    unsigned y;     /* planes y, y + 4 ny, y + 8 ny */
    unsigned list;  /* uint16_t */
    unsigned h;     /* TdFanHead */
    unsigned tab;   /* the team's histogram storage (strip tables, then a part per warp) */
    int ny;
    int T, tw, bar; /* team size, this warp in the team, named barrier */
    int nt;         /* teams of the CTA */
    unsigned part;  /* TdFanPart of the team's first warp, the others TD_WARP_BLOCK_BYTES apart */
};

extern __shared__ __align__(128) unsigned char td_smem[];

template <typename V>
__device__ __forceinline__ V &td_sm(unsigned off)
{
    return *reinterpret_cast<V *>(td_smem + off);
}

__device__ __forceinline__ TdFanHead &td_head(const TdFan &F) { return td_sm<TdFanHead>(F.h); }

__device__ __forceinline__ TdFanPart &td_part(const TdFan &F, int w)
{
    return td_sm<TdFanPart>(F.part + TD_WARP_BLOCK_BYTES * (unsigned)w);
}

/* coordinate r of point pos */
__device__ __forceinline__ float &td_fan_y(const TdFan &F, int r, int pos)
{
    return td_sm<float>(F.y + 4u * (unsigned)(r * F.ny + pos));
}

__device__ __forceinline__ void td_team_sync(const TdFan &F)
{
    if (F.T == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(F.bar), "r"(F.T * 32) : "memory");
}

/* The rows of lane l's minor of the tail: the l-th set of KT rows of D in
 * the order of their bit masks, as a mask (0 past the last). */
template <int D>
__device__ __forceinline__ int td_fan_rowset(int lane)
{
    constexpr int KT = D - 3;
    int seen = 0, mine = 0;
    for (int m = 1; m < (1 << D); ++m)
        if (__popc(m) == KT) {
            if (seen == lane) mine = m;
            ++seen;
        }
    return mine;
}

/* Coefficients of the projection along the tail, by one warp.  P: the KT =
 * K - 1 rows where the tail's minor is largest; for every other row r,
 * F_r(x) = kappa x_r - sum_j d[r][j] x_P[j] with kappa the minor on P and
 * d[r][j] the minor with row P[j] replaced by r (Cramer's rule: on the tail
 * v_r = sum_j (d[r][j] / kappa) v_P[j], so F_r vanishes there).  All exact in
 * int64 (td_coord_limit). */
template <int D>
__device__ __forceinline__ void td_fan_tail(int npc, const int (&c)[D > 2 ? D - 2 : 1], int rowset, float mxall,
                                            unsigned head, int lane)
{
    constexpr int KT = D - 3;
    const float *xs = reinterpret_cast<const float *>(td_smem);
    TdFanHead *h = &td_sm<TdFanHead>(head);
    if (lane == 0) h->mx = 0u;
    if constexpr (KT == 0) {
        if (lane < 3) h->off[4 + lane] = td_xidx(npc, 0, lane);
        if (lane == 0) {
            h->kappa = 1;
            h->mode = 0;
        }
    } else {
        auto minor = [&](const int (&r)[KT]) -> int64_t {
            int32_t m[KT][KT];
#pragma unroll
            for (int a = 0; a < KT; ++a)
#pragma unroll
                for (int b = 0; b < KT; ++b) m[a][b] = td_f2i(xs[td_xidx(npc, c[b + 1], r[a])]);
            if constexpr (KT < 3) {
                return td_detk32<KT>(m); /* 2 max|x|^2 < 2^31 by td_coord_limit */
            } else {
                if (mxall <= 710.f) return td_detk32<KT>(m); /* 6 max|x|^3 < 2^31 */
                int64_t m64[KT][KT];
#pragma unroll
                for (int a = 0; a < KT; ++a)
#pragma unroll
                    for (int b = 0; b < KT; ++b) m64[a][b] = m[a][b];
                return td_detk<KT>(m64);
            }
        };
        auto rows_of = [&](int mask, int (&r)[KT]) {
#pragma unroll
            for (int a = 0; a < KT; ++a) {
                r[a] = mask ? __ffs(mask) - 1 : 0;
                mask &= mask - 1;
            }
        };
        int r[KT];
        rows_of(rowset, r);
        const int64_t P = rowset ? minor(r) : 0;
        const uint32_t key =
            P != 0 ? ((__float_as_uint(fabsf(td_i64_to_f32_bf(P))) & ~31u) | (uint32_t)(31 - lane)) : 0u;
        const uint32_t kmax = __reduce_max_sync(TD_FULL, key);
        if (kmax == 0u) {
            if (lane == 0) h->mode = -1;
            return;
        }
        const int wl = 31 - (int)(kmax & 31u);
        const int64_t kappa = __shfl_sync(TD_FULL, P, wl);
        const int mask = __shfl_sync(TD_FULL, rowset, wl);
        rows_of(mask, r);
        int o[3];
        int rest = ~mask & ((1 << D) - 1);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            o[a] = __ffs(rest) - 1;
            rest &= rest - 1;
        }
        if (lane < 3 * KT) {
            const int ri = lane / KT, j = lane % KT;
            const int orow = ri == 0 ? o[0] : (ri == 1 ? o[1] : o[2]);
            int rr[KT];
#pragma unroll
            for (int a = 0; a < KT; ++a) rr[a] = a == j ? orow : r[a];
            const int64_t v = minor(rr);
            h->d[ri][j] = v;
            h->fd[ri][j] = td_i64_to_f32_bf(v);
        }
        if (lane == 0) {
            h->kappa = kappa;
            h->fk = td_i64_to_f32_bf(kappa);
#pragma unroll
            for (int a = 0; a < KT; ++a) h->off[a] = td_xidx(npc, 0, r[a]);
#pragma unroll
            for (int a = 0; a < 3; ++a) h->off[4 + a] = td_xidx(npc, 0, o[a]);
            /* every |d| <= |kappa| (1 + 2^-17): |kappa| is the largest minor
             * up to the binary32 rounding and the five dropped bits of the
             * key, so K |kappa| max|x| bounds every partial sum of F */
            const float ka = fabsf(td_i64_to_f32_bf(kappa)) * 1.0001f;
            h->mode = (float)(KT + 1) * ka * mxall < 16760000.0f ? 0 : (ka < 2147000000.0f ? 1 : 2);
        }
    }
}

/* Project the points along the tail into the planes; their largest |Y| and
 * the sums of |Y| by coordinate go to the head.  mode 0:
 * every partial sum is an integer below 2^24, exact in binary32; mode 1: the
 * coefficients fit int32, products and sums in int64; mode 2: int64
 * coefficients.  Modes 1 and 2 round Y to binary32 (relative error at most
 * 2u, and a nonzero Y stays nonzero). */
template <int D, int MODE>
__device__ __forceinline__ void td_fan_project_m(int nnz, const TdFan &F, int lane)
{
    constexpr int KT = D - 3;
    const float *xs = reinterpret_cast<const float *>(td_smem);
    const TdFanHead *h = &td_head(F);
    const int npairs = ((nnz + 63) & ~63) >> 1;
    int op[KT > 0 ? KT : 1], oo[3];
    int64_t kap = 1, dd[3][KT > 0 ? KT : 1];
    float fk = 1.f, fd[3][KT > 0 ? KT : 1];
#pragma unroll
    for (int j = 0; j < KT; ++j) op[j] = h->off[j];
#pragma unroll
    for (int r = 0; r < 3; ++r) oo[r] = h->off[4 + r];
    if constexpr (KT > 0) {
        kap = h->kappa;
        fk = h->fk;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < KT; ++j) {
                dd[r][j] = h->d[r][j];
                fd[r][j] = h->fd[r][j];
            }
    }
    unsigned mx = 0u;
    float sum[3] = { 0.f, 0.f, 0.f };
    for (int j0 = 32 * F.tw; j0 < npairs; j0 += 32 * F.T) {
        const int j = j0 + lane; /* npairs is a multiple of 32 */
        float yv[3][2];
        float2 xo[3], xp[KT > 0 ? KT : 1];
#pragma unroll
        for (int r = 0; r < 3; ++r) xo[r] = *reinterpret_cast<const float2 *>(xs + 4 * j + oo[r]);
#pragma unroll
        for (int t = 0; t < KT; ++t) xp[t] = *reinterpret_cast<const float2 *>(xs + 4 * j + op[t]);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if constexpr (KT == 0) {
                yv[r][0] = xo[r].x;
                yv[r][1] = xo[r].y;
            } else if constexpr (MODE == 0) {
                float a = fk * xo[r].x, b = fk * xo[r].y;
#pragma unroll
                for (int t = 0; t < KT; ++t) {
                    a = fmaf(-fd[r][t], xp[t].x, a);
                    b = fmaf(-fd[r][t], xp[t].y, b);
                }
                yv[r][0] = a;
                yv[r][1] = b;
            } else {
                int64_t a, b;
                if constexpr (MODE == 1) {
                    a = (int64_t)(int32_t)kap * td_f2i(xo[r].x);
                    b = (int64_t)(int32_t)kap * td_f2i(xo[r].y);
                } else {
                    a = kap * td_f2i(xo[r].x);
                    b = kap * td_f2i(xo[r].y);
                }
#pragma unroll
                for (int t = 0; t < KT; ++t) {
                    if constexpr (MODE == 1) {
                        a -= (int64_t)(int32_t)dd[r][t] * td_f2i(xp[t].x);
                        b -= (int64_t)(int32_t)dd[r][t] * td_f2i(xp[t].y);
                    } else {
                        a -= dd[r][t] * td_f2i(xp[t].x);
                        b -= dd[r][t] * td_f2i(xp[t].y);
                    }
                }
                yv[r][0] = td_i64_to_f32_bf(a);
                yv[r][1] = td_i64_to_f32_bf(b);
            }
            sum[r] += fabsf(yv[r][0]) + fabsf(yv[r][1]);
            mx = max(mx, max(__float_as_uint(yv[r][0]) & 0x7fffffffu, __float_as_uint(yv[r][1]) & 0x7fffffffu));
        }
        const int i = 2 * j0 + lane; /* points i and i + 32; the planes end after a multiple of 32 */
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            td_fan_y(F, r, i) = yv[r][0];
            if (2 * j0 + 32 < F.ny) td_fan_y(F, r, i + 32) = yv[r][1];
        }
    }
    mx = __reduce_max_sync(TD_FULL, mx);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum[r] += __shfl_xor_sync(TD_FULL, sum[r], o);
    if (lane == 0) {
        atomicMax(&td_head(F).mx, mx);
#pragma unroll
        for (int r = 0; r < 3; ++r) td_part(F, F.tw).sum[r] = sum[r];
    }
}

/* ---- bounds of all subsets of a fan at once -------------------------------
 * Directions v = (cos, sin, -tau) of the fan's 3-D quotient, the angle of
 * (cos, sin) in [0, pi): the count of a halfspace is f(v) = #{ i : v.Y_i < 0 },
 * and with A_i = Y_i0 / Y_i2, B_i = Y_i1 / Y_i2 (each coordinate scaled to the
 * same mean size first) the sign of v.Y_i is that of Y_i2 (t_i - tau), t_i =
 * A_i cos + B_i sin.  The subset of c_0 has the directions tau = t_c0, so its
 * walk is f along the curve t_c0, and a point whose curve stays on one side of
 * t_c0 keeps its sign.  The half turn is cut into K strips between the
 * directions d_k = (cos, sin)(pi k / K); inside a strip directions are taken
 * as (1 - l) d_k + l d_(k+1), where every t_i is linear in l and lies between
 * its two end values.  So with the range [lo_i, hi_i] of bins of the key t /
 * (1 + |t|) at the two ends, a point of hi_i < lo_c is below the curve of c
 * throughout the strip, and one of lo_i > hi_c above it.  Their numbers, split
 * by the sign of Y_i2, are two prefix sums of a histogram: for every c
 *
 *     f >= #{ below, + } + #{ above, - },  n - f >= #{ above, + } + #{ below, - }
 *
 * in the strip, and the smaller value over all strips bounds G(c) from below.
 * Only the points' ranges need to be whole: the curve of c is cut into two
 * pieces of half its range of bins each, bounded one by one (in a simulation
 * of the p = 5 data set with ties 8 strips then leave 0.5% of the subsets to
 * the quads, against 3.8% with one piece; with four pieces it is 0.1%, but
 * the look-ups cost more than that saves: 36.8 ms against 33.9, and 36.5 with
 * one).
 * It counts every point, as the sweep's row histogram does, but costs a
 * number of steps per strip and point of the fan instead of per point and
 * subset.  Subsets whose bound reaches best in every strip are done.
 *
 * Rounding: A and B have relative errors below 8.2u (Y 2u each, reciprocal
 * 2u, two products), so t is off by less than 10.3u (|A| + |B|), and the key by
 * less than that plus 3.1u; for |A| + |B| <= 2048 and at most 256 bins (of
 * width 1/128) that is below 0.17 of a bin.  So hi_i + 2 <= lo_c fixes the
 * order.  Points beyond 2048, or with Y_2 = 0, are counted nowhere (as c:
 * never done here). */
__device__ __forceinline__ int td_strip_key(float A, float B, float2 d, float M)
{
    const float t = fmaf(B, d.y, A * d.x);
    return __float_as_int(__fmaf_rd(t, td_rcp(1.0f + fabsf(t)), M)); /* bits(M) + floor(key bins / 2) */
}

/* KC strips at a time (what the team's histogram storage holds), NB bins.
 * 256 bins where rows are long: the two bins that an order needs between two
 * points are 2 n / NB of them.  128 and the byte-packed form for at most 255
 * points: half the tables to clear and to sum, twice the strips a round; 256
 * bins there made p = 5, n = 200 36.9 ms against 32.9.  512 bins, 4 strips at a
 * time, made W2 4.1 ms against 3.4.  Returns the lanes' flags: bit it of a
 * lane is set when the subset of point 32 (tw + T it) + lane is left. */
template <int KC, int NB, bool PACKED>
__device__ __forceinline__ uint32_t td_fan_strips(int nnz, const TdFan &F, int lo, int hi, int K, const float2 *dirs,
                                                  int best, int lane)
{
    constexpr int WORDS = TD_STRIP_WORDS(NB, PACKED), LB = NB == 256 ? 8 : 7;
    constexpr int GW = PACKED ? 0 : NB;         /* words from the upper ends' bins to the lower ends' */
    constexpr int NA = PACKED ? KC : 2 * KC;    /* arrays */
    static_assert(NB == 256 || NB == 128, "bins");
    constexpr unsigned MB = ((unsigned)(127 + 24 - LB) << 23) | 0x400000u; /* M = 1.5 * 2^(24 - LB): spacing 2 / NB */
    const float M = __uint_as_float(MB);
    const int T = F.T, st = TD_STRIP_MAX / K; /* dirs holds TD_STRIP_MAX + 1 directions */
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    for (int w = 0; w < T; ++w) {
        s0 += td_part(F, w).sum[0];
        s1 += td_part(F, w).sum[1];
        s2 += td_part(F, w).sum[2];
    }
    /* scales; a coordinate that vanishes throughout leaves no usable ratio */
    const float g0 = s0 > 0.f ? s2 * td_rcp(s0) : 0.f, g1 = s1 > 0.f ? s2 * td_rcp(s1) : 0.f;
    auto ratios = [&](int pos, float &A, float &B, float &h) -> bool {
        const float y0 = td_fan_y(F, 0, pos), y1 = td_fan_y(F, 1, pos);
        h = td_fan_y(F, 2, pos);
        const float r = td_rcp(h);
        A = y0 * (g0 * r);
        B = y1 * (g1 * r);
        const bool ok = h != 0.f && fabsf(A) + fabsf(B) <= 2048.f; /* false for NaN */
        if (!ok) A = B = 0.f;
        return ok;
    };
    /* byte address of a key's bin in the first strip's table, less 4 key */
    const unsigned tb = td_saddr(td_smem) + F.tab + 16u + 4u * (NB / 2) - 4u * MB;
    uint32_t fail = 0u;
    const int b16 = min(best, 0x7fff);
    const uint32_t bias0 = (uint32_t)(0x8000 - b16) * 0x10001u;
    for (int k0 = 0; k0 < K; k0 += KC) {
        if (k0 > 0) td_team_sync(F); /* the previous tables are read */
        for (int j = 32 * F.tw + lane; j < KC * WORDS / 4; j += 32 * T)
            td_sm<uint4>(F.tab + 16u * (unsigned)j) = make_uint4(0u, 0u, 0u, 0u);
        td_team_sync(F);
        const float2 *dk = dirs + k0 * st;
        for (int p0 = 32 * F.tw; p0 < nnz; p0 += 32 * T) {
            const int pos = p0 + lane; /* below ny: the planes are padded with zeros */
            float A, B, h;
            const uint32_t inc = ratios(pos, A, B, h) ? (h > 0.f ? 1u : (PACKED ? 0x100u : 0x10000u)) : 0u;
            const uint32_t incg = PACKED ? inc << 16 : inc;
            int v = td_strip_key(A, B, dk[0], M);
            const float2 *d = dk;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int v2 = td_strip_key(A, B, *(d += st), M);
                td_reds_add(tb + 4u * (unsigned)max(v, v2) + 4u * WORDS * k, inc);
                td_reds_add(tb + 4u * (unsigned)min(v, v2) + 4u * (WORDS * k + GW), incg);
                v = v2;
            }
        }
        td_team_sync(F);
        /* prefix sums of every array (packed counts of the two signs, of
         * both ends if PACKED), the total after the last bin; the warps
         * share the arrays, four at a time so that their scans overlap */
        for (int a0 = 4 * F.tw; a0 < NA; a0 += 4 * T) {
            constexpr int Q = NB / 128; /* quads per lane */
            uint4 q[4][Q];
            uint32_t sum[4], inc[4];
            unsigned t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int a = a0 + u;
                t[u] = F.tab + 4u * (unsigned)(PACKED ? a * WORDS + 4 : (a >> 1) * WORDS + 4 + (a & 1) * NB);
                sum[u] = 0u;
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    q[u][j] = td_sm<uint4>(t[u] + 16u * (unsigned)(Q * lane + j));
                    q[u][j].x += sum[u];
                    q[u][j].y += q[u][j].x;
                    q[u][j].z += q[u][j].y;
                    q[u][j].w += q[u][j].z;
                    sum[u] = q[u][j].w;
                }
                inc[u] = sum[u];
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t x = __shfl_up_sync(TD_FULL, inc[u], o);
                    if (lane >= o) inc[u] += x;
                }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t ex = inc[u] - sum[u];
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    q[u][j].x += ex;
                    q[u][j].y += ex;
                    q[u][j].z += ex;
                    q[u][j].w += ex;
                    td_sm<uint4>(t[u] + 16u * (unsigned)(Q * lane + j)) = q[u][j];
                }
                /* (unpacked: the words after an upper-end array belong to
                 * the lower-end one) */
                if (lane == 31 && (PACKED || (u & 1))) td_sm<uint32_t>(t[u] + 4u * NB) = inc[u];
            }
        }
        td_team_sync(F);
        /* every strip's total is that of the counted points, by sign */
        const uint32_t total = td_sm<uint32_t>(F.tab + 4u * (4 + GW + NB));
        const uint32_t bias = __byte_perm(total, 0u, PACKED ? 0x4243 : 0x1032) + bias0;
        int it = 0;
        for (int p0 = 32 * F.tw; p0 < hi; p0 += 32 * T, ++it) {
            if (p0 + 32 <= lo) continue; /* no value of c_0 in this block */
            const int pos = p0 + lane;
            float A, B, h;
            uint32_t acc = ratios(pos, A, B, h) ? 0x80008000u : 0u;
            int v = td_strip_key(A, B, dk[0], M);
            const float2 *d = dk;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int v2 = td_strip_key(A, B, *(d += st), M);
                /* both halves of the curve's range of bins, each with the
                 * points below its lower and above its upper end.  Low half
                 * of a word: below and + with above and -; high half: the
                 * others; bit 15 of a half says that it reaches best. */
                const int x0 = min(v, v2), x2 = max(v, v2), x1 = td_key_middle(x0, x2);
                const uint32_t f0 = td_lds32(tb + 4u * (unsigned)x0 + 4u * (WORDS * k - 2));
                const uint32_t g0 = td_lds32(tb + 4u * (unsigned)x1 + 4u * (WORDS * k + GW + 1));
                const uint32_t f1 = td_lds32(tb + 4u * (unsigned)x1 + 4u * (WORDS * k - 2));
                const uint32_t g1 = td_lds32(tb + 4u * (unsigned)x2 + 4u * (WORDS * k + GW + 1));
                if (PACKED) {
                    acc &= __byte_perm(f0, 0u, 0x4140) - __byte_perm(g0, 0u, 0x4243) + bias;
                    acc &= __byte_perm(f1, 0u, 0x4140) - __byte_perm(g1, 0u, 0x4243) + bias;
                } else {
                    acc &= f0 - __byte_perm(g0, 0u, 0x1032) + bias;
                    acc &= f1 - __byte_perm(g1, 0u, 0x1032) + bias;
                }
                v = v2;
            }
            if (acc != 0x80008000u) fail |= 1u << it;
        }
    }
    return fail;
}

/* Subsets to sweep one by one: the c_0 values lo <= i < hi whose bit is set in
 * the lanes' flags (bit it of a lane: point 32 (tw + T it) + lane), and the
 * dependent ones (Y = 0, whose flag is always set). */
__device__ __forceinline__ bool td_fan_flag(const TdFan &F, int i, int lo, int hi, uint32_t fail, int it, bool &zero)
{
    const bool flag = i >= lo && i < hi && ((fail >> it) & 1u);
    zero = false;
    if (__any_sync(TD_FULL, flag))
        zero = flag && td_fan_y(F, 0, i) == 0.f && td_fan_y(F, 1, i) == 0.f && td_fan_y(F, 2, i) == 0.f;
    return flag && !zero;
}

__device__ __forceinline__ void td_fan_count(const TdFan &F, int lo, int hi, uint32_t fail, int lane)
{
    int n = 0, dep = 0, it = 0;
    for (int p0 = 32 * F.tw; p0 < hi; p0 += 32 * F.T, ++it) {
        bool zero;
        n += __popc(__ballot_sync(TD_FULL, td_fan_flag(F, p0 + lane, lo, hi, fail, it, zero)));
        dep += __popc(__ballot_sync(TD_FULL, zero));
    }
    if (lane == 0) {
        td_part(F, F.tw).left = n;
        td_part(F, F.tw).dependent = dep;
    }
}

/* Their list, in increasing order per warp. */
__device__ __forceinline__ void td_fan_list(const TdFan &F, int lo, int hi, uint32_t fail, int lane)
{
    int o = 0, it = 0;
    for (int w = 0; w < F.tw; ++w) o += td_part(F, w).left;
    for (int p0 = 32 * F.tw; p0 < hi; p0 += 32 * F.T, ++it) {
        bool zero;
        const bool mine = td_fan_flag(F, p0 + lane, lo, hi, fail, it, zero);
        const unsigned b = __ballot_sync(TD_FULL, mine);
        if (mine) td_sm<uint16_t>(F.list + 2u * (unsigned)(o + __popc(b & ((1u << lane) - 1u)))) = (uint16_t)(p0 + lane);
        o += __popc(b);
    }
}

/* Constants of a quad's point loop. */
struct TdFanConst {
    td_f2x c, nc; /* (+c, +c), (-c, -c): half width of the direction interval */
    td_f2x km;    /* (M + 1, M + 1), M = 1.5 * 2^16: binary32 spacing 1/128 */
};

/* bits(M): the row is the bit pattern less this */
#define TD_FAN_MBITS 0x47C00000u

/* One staged pair of points against one subset: both events to the subset's
 * table at byte offset OFF from tb.
 *
 * Certification.  kappa = U1 sgn(U2) / (|U1| + |U2|) in [-1, 1] decreases with
 * the angle of the line direction; the rows are floor((kappa + 1) 128) (the
 * sweep in the mirrored order, which has the same walk values).  With
 * E >= |u - U| for both computed coordinates and s = |u1| + |u2| > 4E,
 * kappa changes by at most E / (s - 2E) <= 2E / s between u and U while U2
 * keeps its sign.  The two ends are rr (u1 +- c) with rr the approximate
 * reciprocal of s signed as u2 (sum, reciprocal and u1 +- c: relative errors
 * u, 2u, u), and the directed multiply-add with M + 1 is an exact floor of
 * rr (u1 +- c) + 1 on the grid 1/128.  So the ends enclose kappa +- 2E / s
 * when c (1 - 4.1u) >= 2E + 4.1u s; s <= 4.01 X for X = max |Y| (both ratios
 * are at most 1), and E = 14u X (below), hence c = 48u X.  Equal ends then
 * fix the row; which of the two is the upper one does not matter.  They also
 * fix the sign of U2: it can be wrong only if |u2| <= E, then
 * |kappa| >= 1 - E / s and the outer end passes +-1 by E / s: the floors
 * differ.  Both ends outside [-1, 1) on one side is impossible (|u1 rr| <=
 * 1 + 3u, c |rr| > 10u).  For s <= 4E the ends are more than 1.7 apart, and
 * for s = 0 (the subset's own points, padding) they are +-infinity.
 *
 * E: |Y_f - Y| <= 2u |Y|, the ratio of two such values through the
 * approximate reciprocal (2u) and a product has error at most 7.1u (it is at
 * most 1), the multiply-add rounds once (u 2X): u (2 + 2 + 7.1 + 2.1) X < 14u X.
 *
 * An uncertain point goes to the row that is not read: their count is the number of points less
 * the events found in the table.  The event's word is 0x10000 plus the sign
 * bit of u2 (high half: events, low half: +1 events). */
template <int OFF>
__device__ __forceinline__ void td_fan_pair(td_f2x ya, td_f2x yb, td_f2x yp, td_f2x na, td_f2x nb,
                                            const TdFanConst &C, unsigned tb)
{
    const td_f2x U1 = td_fma2(na, yp, ya), U2 = td_fma2(nb, yp, yb);
    float u1p, u1q, u2p, u2q;
    td_upk(U1, u1p, u1q);
    td_upk(U2, u2p, u2q);
    const td_f2x S = td_add2(U2, td_pk(copysignf(u1p, u2p), copysignf(u1q, u2q))); /* |u1| + |u2|, signed as u2 */
    float sp, sq;
    td_upk(S, sp, sq);
    const td_f2x RR = td_pk(td_rcp(sp), td_rcp(sq));
    const td_f2x FA = td_fma2_rm(RR, td_add2(U1, C.c), C.km);
    const td_f2x FB = td_fma2_rm(RR, td_add2(U1, C.nc), C.km);
    float fap, faq, fbp, fbq;
    td_upk(FA, fap, faq);
    td_upk(FB, fbp, fbq);
    const unsigned rp = __float_as_int(fap) == __float_as_int(fbp) ? (unsigned)__float_as_int(fap) : TD_FAN_MBITS + TD_FAN_ROWS;
    const unsigned rq = __float_as_int(faq) == __float_as_int(fbq) ? (unsigned)__float_as_int(faq) : TD_FAN_MBITS + TD_FAN_ROWS;
    td_reds_at<OFF>(tb + (rp << 2), 0x10000u + ((unsigned)__float_as_int(u2p) >> 31));
    td_reds_at<OFF>(tb + (rq << 2), 0x10000u + ((unsigned)__float_as_int(u2q) >> 31));
}

/* The query's running minimum, which other warps lower at any time, as lane 0
 * read it last.  What is decided from it guards full-warp operations, so every
 * lane takes that one value: loads of 32 lanes that have come apart (after a
 * block of lane 0 alone, say) may see different ones.  read() one step ahead
 * of its get(): the wait for the load is hidden, the shuffle is not seen. */
struct TdQmin {
    int v;
    __device__ __forceinline__ void read(const int32_t *qmin) { v = *reinterpret_cast<const volatile int32_t *>(qmin); }
    __device__ __forceinline__ int get() const { return __shfl_sync(TD_FULL, v, 0); }
};

/* ---- four subsets in one pass ------------------------------------------
 * In the 3-D coordinates Y of the fan the subset of c_0 projects by
 *
 *     U1 = Y_a - (Y_a(c_0) / Y_p(c_0)) Y_p,   U2 = Y_b - (Y_b(c_0) / Y_p(c_0)) Y_p
 *
 * with p the coordinate where |Y(c_0)| is largest and (p, a, b) cyclic: two
 * multiply-adds a point instead of 2 D, and a basis that is one reciprocal and
 * two products.  U is a linear isomorphism of the quotient R^D / span(S) onto
 * R^2 (both functionals vanish on S and they are independent), and the
 * bivariate depth of the origin does not depend on which one is used.
 *
 * The events of nv <= 4 subsets, into the warp's tables.  oa, ob, op: byte
 * offsets (from the planes' start) of the planes a, b, p of each subset.  Full
 * blocks of 64 points take a pair a lane and subset; the last partial block,
 * when it holds at most 48 points, is spread over the four subsets instead:
 * lanes 8 g .. 8 g + 7 place 16 points of subset g a step. */
__device__ __forceinline__ void td_fan_points(unsigned ybase, int nnz, int nv, int lane, const unsigned (&oa)[4],
                                              const unsigned (&ob)[4], const unsigned (&op)[4], unsigned coef,
                                              const TdFanConst &C, unsigned tab)
{
    td_f2x na[4], nb[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) td_lds_coef(coef + 16u * s, na[s], nb[s]);
    const unsigned tb = tab - (TD_FAN_MBITS << 2);
    const int rem = nnz & 63;
    const int end = rem > 48 ? nnz + 64 - rem : nnz - rem;
    unsigned a = ybase + 8u * (unsigned)lane;
    const unsigned ae = ybase + 4u * (unsigned)end;
    for (; a < ae; a += 256u) {
        td_fan_pair<0>(td_lds64(a + oa[0]), td_lds64(a + ob[0]), td_lds64(a + op[0]), na[0], nb[0], C, tb);
        if (nv > 1)
            td_fan_pair<TD_FAN_TABLE>(td_lds64(a + oa[1]), td_lds64(a + ob[1]), td_lds64(a + op[1]), na[1], nb[1], C, tb);
        if (nv > 2)
            td_fan_pair<2 * TD_FAN_TABLE>(td_lds64(a + oa[2]), td_lds64(a + ob[2]), td_lds64(a + op[2]), na[2], nb[2], C, tb);
        if (nv > 3)
            td_fan_pair<3 * TD_FAN_TABLE>(td_lds64(a + oa[3]), td_lds64(a + ob[3]), td_lds64(a + op[3]), na[3], nb[3], C, tb);
    }
    if (rem > 0 && rem <= 48) {
        const int g = lane >> 3;
        td_f2x ng, mg;
        td_lds_coef(coef + 16u * (unsigned)g, ng, mg);
        unsigned ga = oa[0], gb = ob[0], gp = op[0];
#pragma unroll
        for (int s = 1; s < 4; ++s)
            if (g == s) {
                ga = oa[s];
                gb = ob[s];
                gp = op[s];
            }
        const unsigned tg = tb + (unsigned)g * TD_FAN_TABLE;
        unsigned b = ybase + 4u * (unsigned)(nnz - rem) + 8u * (unsigned)(lane & 7);
        for (int k = 0; k < rem; k += 16, b += 64u)
            td_fan_pair<0>(td_lds64(b + ga), td_lds64(b + gb), td_lds64(b + gp), ng, mg, C, tg);
    }
}

/* Subsets list[first .. first + nv) of the fan (nv <= 4; c[1..K) its tail):
 * bounds from one pass over the points and 256 angular rows each, then the
 * exact sweep of those that do not reach best. */
template <int D>
__device__ __forceinline__ void td_fan_quad(const TdLaunch &L, int q, int nnz, const TdFan &F, int first, int nv,
                                            const int (&c)[D - 2], unsigned wb, unsigned mb, int lane, int &best)
{
    constexpr int K = D - 2;
    /* lane s < 4: subset s of the quad (past the end: subset 0 again) */
    const int s = lane & 3;
    const int i = td_sm<uint16_t>(F.list + 2u * (unsigned)(first + (s < nv ? s : 0)));
    const float v0 = td_fan_y(F, 0, i), v1 = td_fan_y(F, 1, i), v2 = td_fan_y(F, 2, i);
    const float a0 = fabsf(v0), a1 = fabsf(v1), a2 = fabsf(v2);
    const int k = a0 >= a1 ? (a0 >= a2 ? 0 : 2) : (a1 >= a2 ? 1 : 2);
    const float yp = k == 0 ? v0 : (k == 1 ? v1 : v2);
    const float ya = k == 0 ? v1 : (k == 1 ? v2 : v0);
    const float yb = k == 0 ? v2 : (k == 1 ? v0 : v1);
    const float r = -td_rcp(yp);
    const unsigned co = mb + 16u + 192u; /* the basis block's packed columns */
    __syncwarp(); /* the coefficients and the tables of the previous quad are read */
    if (lane < 4) {
        const float na = ya * r, nb = yb * r;
        td_sm<float4>(co + 16u * (unsigned)lane) = make_float4(na, na, nb, nb);
    }
    for (int j = lane; j < (4 * TD_FAN_TABLE >> 4); j += 32) td_sm<uint4>(wb + 16u * (unsigned)j) = make_uint4(0u, 0u, 0u, 0u);
    TdFanConst C;
    {
        const float cw = 48.0f * TD_U * __uint_as_float(td_head(F).mx), M1 = 98305.0f; /* 1.5 * 2^16 + 1 */
        C.c = td_pk(cw, cw);
        C.nc = td_pk(-cw, -cw);
        C.km = td_pk(M1, M1);
    }
    __syncwarp();
    const unsigned pl = 4u * (unsigned)F.ny;
    const unsigned sb = td_saddr(td_smem), ybase = sb + F.y, tab = sb + wb, coef = sb + co;
    unsigned oa[4], ob[4], op[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int kt = __shfl_sync(TD_FULL, k, t);
        op[t] = kt == 0 ? 0u : (kt == 1 ? pl : 2u * pl);
        oa[t] = kt == 0 ? pl : (kt == 1 ? 2u * pl : 0u);
        ob[t] = kt == 0 ? 2u * pl : (kt == 1 ? 0u : pl);
    }
    td_fan_points(ybase, nnz, nv, lane, oa, ob, op, coef, C, tab);
    __syncwarp();
    /* Pass 1: lane l scans rows 8 l .. 8 l + 7 of each table.  In a row the
     * walk stays within [P - cm, P + cp]; over the certified points only,
     * min(w, nc - w) is a lower bound (see td_sweep_filtered). */
    int mylb = INT_MAX; /* lane t: the bound of subset t */
    bool low = false;
    int ncs = 0; /* certified points */
#pragma unroll 1
    for (int t = 0; t < nv; ++t) {
        const unsigned h4 = wb + (unsigned)(t * TD_FAN_TABLE + 32 * lane);
        const uint4 qa = td_sm<uint4>(h4), qb = td_sm<uint4>(h4 + 16u);
        const uint32_t w8[8] = { qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w };
        uint32_t sum = 0;
        int P = 0, lom = 0, him = 0; /* walk relative to the lane's start, the extremes of its bounds */
        int lob = 0, hib = 0;        /* and of the walk at the row boundaries */
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int cp = td_ev_plus(w8[j]), cm = td_ev_minus(w8[j]);
            sum += w8[j];
            lom = min(lom, P - cm);
            him = max(him, P + cp);
            P += cp - cm;
            lob = min(lob, P);
            hib = max(hib, P);
        }
        const int cp = td_ev_plus(sum), cm = td_ev_minus(sum);
        const int A = td_wsum(cm); /* orientation + points */
        const int nc = A + td_wsum(cp);
        const int ex = td_wscan_incl(cp - cm, lane) - (cp - cm);
        const int val = min(A + ex + lom, nc - (A + ex + him));
        const int lb = td_wmin(val);
        if (lane == t) mylb = lb;
        ncs += nc;
        if (lb < best) {
            low = true;
            /* At a row boundary the certified points are on known sides: the
             * walk value there plus all others is a halfspace count, so it
             * is not below V(S), and best may take it */
            const int ub = td_wmin(min(A + ex + lob, nc - (A + ex + hib))) + nnz - nc;
            if (ub < best) {
                best = ub;
                if (lane == 0) atomicMin(L.qmin + q, ub);
            }
        }
    }
    if (lane == 0) {
        unsigned long long *ws = td_warp_stats(mb);
        ws[2] += (unsigned)ncs;
        ws[3] += (unsigned)(nv * nnz - ncs);
    }
    if (low) {
#pragma unroll 1
        for (int t = 0; t < nv; ++t) {
            if (__shfl_sync(TD_FULL, mylb, t) >= best) continue;
            const int it = __shfl_sync(TD_FULL, i, t);
            const int V = td_sweep_one<D>(&L, q, nnz, it, K > 1 ? c[K > 1 ? 1 : 0] : 0, K > 2 ? c[K > 2 ? 2 : 0] : 0, K > 3 ? c[K > 3 ? 3 : 0] : 0, wb, mb, best);
            if (V < best) {
                best = V;
                if (lane == 0) atomicMin(L.qmin + q, V);
            }
        }
    }
}

/* How a team bounds its fans.  k: strips.  Their cost is about k (12 nnz + 15 m
 * + 2000) / 32 warp instructions for a fan of m values of c_0, and every subset
 * they leave costs about (11 nnz + 1600) / 32 in a quad; k doubles while the
 * quads cost more than the strips and halves when they cost less than a
 * sixth.  rest: fans to go without strips, because even the most strips left
 * more than half of the subsets (points on few lines, say). */
struct TdFanPlan {
    int k, rest;
};

__device__ __forceinline__ int td_fan_choose(TdFanPlan &P, int nnz, int m)
{
    if (P.rest > 0) {
        --P.rest;
        return 0;
    }
    return 5 * P.k * (12 * nnz + 15 * m + 2000) < 4 * m * (11 * nnz + 1600) ? P.k : 0;
}

__device__ __forceinline__ void td_fan_learn(TdFanPlan &P, int nnz, int m, int left)
{
    const int strips = P.k * (12 * nnz + 15 * m + 2000), quads = left * (11 * nnz + 1600);
    if (quads > strips) {
        if (P.k < TD_STRIP_MAX) P.k *= 2;
        else if (2 * left > m) P.rest = 7;
    } else if (6 * quads < strips && P.k > 8) {
        P.k /= 2;
    }
}

/* The fans of subset positions [r0, r0 + count) of query q that this team
 * takes: the tile's fans are numbered in order and taken from the counter
 * *ticket (the first ones: the team's own number).  wb, mb: this warp's
 * histogram storage and basis block. */
template <int D>
__device__ __forceinline__ void td_team_sweep(const TdLaunch &L, int q, int nnz, uint64_t r0, int count, int mine,
                                              int *ticket, const TdFan &F, TdFanPlan &P, unsigned wb, unsigned mb,
                                              const float2 *dirs, int rowset, int lane, int &best)
{
    constexpr int K = D - 2;
    if (count <= 0) return;
    int c[K];
    td_unrank_colex<K>(r0, nnz, c);
    float mxall = 0.f;
#pragma unroll
    for (int r = 0; r < D; ++r) mxall = fmaxf(mxall, (float)L.q[q].mx[r]); /* < 2^22: exact */
    TdQmin gbest = { best };
    if (F.tw == 0 && lane == 0) td_head(F).stop = 0;
    td_team_sync(F);
    for (int fan = 0; count > 0; ++fan) {
        const int lo = c[0];
        const int m = K >= 2 ? min(count, c[K >= 2 ? 1 : 0] - lo) : count, hi = lo + m;
        if (fan == mine) {
            const bool stop = L.early_exit && td_head(F).stop; /* written before the last barrier only */
            if (F.tw == 0) {
                if (!stop) td_fan_tail<D>(td_plane_pairs(L.nmax), c, rowset, mxall, F.h, lane);
                if (lane == 0) td_head(F).next = F.nt + atomicAdd(ticket, 1);
            }
            best = min(best, gbest.get());
            gbest.read(L.qmin + q);
            td_team_sync(F);
            mine = td_head(F).next;
            const int mode = stop ? -2 : td_head(F).mode;
            if (mode >= 0) {
                if (mode == 0) td_fan_project_m<D, 0>(nnz, F, lane);
                else if (mode == 1) td_fan_project_m<D, 1>(nnz, F, lane);
                else td_fan_project_m<D, 2>(nnz, F, lane);
                td_team_sync(F);
                const int ks = td_fan_choose(P, nnz, m);
                uint32_t fail = 0xffffffffu;
                if (ks > 0)
                    fail = F.T > 2      ? td_fan_strips<8, 256, false>(nnz, F, lo, hi, ks, dirs, best, lane)
                           : F.T == 2   ? td_fan_strips<4, 256, false>(nnz, F, lo, hi, ks, dirs, best, lane)
                           : nnz <= 255 ? td_fan_strips<8, 128, true>(nnz, F, lo, hi, ks, dirs, best, lane)
                                        : td_fan_strips<4, 128, false>(nnz, F, lo, hi, ks, dirs, best, lane);
                td_fan_count(F, lo, hi, fail, lane);
                td_team_sync(F);
                int ntot = 0, nd = 0;
                for (int w = 0; w < F.T; ++w) {
                    ntot += td_part(F, w).left;
                    nd += td_part(F, w).dependent;
                }
                if (F.tw == 0 && lane == 0) {
                    unsigned long long *ws = td_warp_stats(mb);
                    ws[0] += (unsigned)(m - nd);
                    ws[1] += (unsigned)nd;
                }
                if (ks > 0) td_fan_learn(P, nnz, m, ntot);
                if (ntot > 0) {
                    td_fan_list(F, lo, hi, fail, lane);
                    td_team_sync(F);
                    /* fewer than four a warp when they are few, so that every
                     * warp has some */
                    const int gs = min(4, (ntot + F.T - 1) / F.T);
                    for (int g = gs * F.tw; g < ntot; g += gs * F.T) {
                        /* the query's minimum, lowered by other warps: read
                         * one quad ahead of its use */
                        best = min(best, gbest.get());
                        gbest.read(L.qmin + q);
                        if (L.early_exit && best <= 0) {
                            /* V = 0 is the least value: nothing can lower it */
                            const unsigned long long left = (unsigned)min(gs, ntot - g);
                            if (lane == 0) {
                                unsigned long long *ws = td_warp_stats(mb);
                                ws[0] -= left;
                                ws[7] += left;
                            }
                            continue;
                        }
                        td_fan_quad<D>(L, q, nnz, F, g, min(gs, ntot - g), c, wb, mb, lane, best);
                    }
                }
                if (L.early_exit && best <= 0 && lane == 0) td_head(F).stop = 1;
            } else if (F.tw == 0 && lane == 0) {
                td_warp_stats(mb)[stop ? 7 : 1] += (unsigned)m;
            }
            td_team_sync(F); /* the planes, the list, the tables and the head are rewritten next */
        }
        count -= m;
        if (K >= 2 && count > 0) {
            c[0] = hi - 1;
            td_next_colex<K>(c);
        }
    }
    best = min(best, gbest.get());
}
