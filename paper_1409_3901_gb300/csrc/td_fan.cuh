/*
 * td_fan.cuh -- the filtered sweep for effective dimensions D = 3 .. 6: four
 * subsets that share all points but one in one pass over the data.
 *
 * Consecutive colex positions S = {c_0 < c_1 < .. < c_(K-1)} (K = D - 2)
 * share the tail (c_1, .., c_(K-1)) while c_0 runs from 0 to c_1 - 1; such a
 * run is called a fan.  Projecting along span(S) can be done in two steps:
 * first along the tail, R^D -> R^3, once for the fan (exact integers), then
 * along the one remaining point, R^3 -> R^2, for every subset.  In the 3-D
 * coordinates Y the second step is
 *
 *     U1 = Y_a - (Y_a(c_0) / Y_p(c_0)) Y_p,   U2 = Y_b - (Y_b(c_0) / Y_p(c_0)) Y_p
 *
 * with p the coordinate where |Y(c_0)| is largest and (p, a, b) cyclic: two
 * multiply-adds a point instead of 2 D, and a basis that is one reciprocal and
 * two products instead of C(D, 2) minors of order K, their maximum and their
 * shuffles.  U is a linear isomorphism of the quotient R^D / span(S) onto R^2
 * (both functionals vanish on S and they are independent), and the bivariate
 * depth of the origin does not depend on which isomorphism is used.
 *
 * A team of T warps (T a power of two dividing the CTA) takes a fan: it
 * projects the points along the tail into shared memory, sorts the values of
 * c_0 by their pivot coordinate p, and its warps take four subsets of one
 * pivot at a time (td_fan_quad).  A subset whose lower bound does not reach
 * the running minimum is swept again alone with the exact steps
 * (td_sweep_one); the others are done.
 */
#pragma once

/* Rows of a quad's histograms: 256 per subset, plus one word that takes the
 * uncertain points (never read: a store to it costs less than a branch around
 * it).  Bytes per subset, a multiple of 16. */
#define TD_FAN_ROWS 256
#define TD_FAN_TABLE ((TD_FAN_ROWS + 4) * 4)

/* Strip tables (td_fan_strips): words per strip (4 of padding, the bins of
 * the upper ends, the bins of the lower ends, 4 of padding).  A team's
 * histogram storage, TD_FAN_HIST bytes or more per warp, holds 4 strips of
 * 128 bins for one warp, 8 for two, and 8 of 256 bins for more. */
#define TD_STRIP_WORDS(bins) (2 * (bins) + 8)
#define TD_STRIP_MAX 64 /* strips, at most */
#define TD_FAN_HIST (4 * TD_STRIP_WORDS(128) * 4)
static_assert(TD_FAN_HIST % 128 == 0 && 2 * TD_STRIP_WORDS(256) * 4 <= TD_FAN_HIST && 4 * TD_FAN_TABLE <= TD_FAN_HIST,
              "warp histogram storage");

#ifndef TD_FAN_SPREAD
#define TD_FAN_SPREAD 96
#endif
#ifndef TD_STRIP_FIRST
#define TD_STRIP_FIRST 16
#endif

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

/* Warps per team for rows of nnz points: the mean fan holds about nnz /
 * (D - 1) subsets (nnz / 2 at D = 4, nnz / 3 at D = 5), and a team meets at
 * barriers around each fan, so every warp should get at least about eight
 * quads of it.  At D = 3 the whole tile is one fan. */
__host__ __device__ inline int td_fan_team(int D, int nnz, int warps)
{
    if (D == 3) return warps;
    int t = 1;
    while (2 * t <= warps && 2 * t * TD_FAN_SPREAD * (D - 2) <= nnz) t *= 2;
    return t;
}

/* A team's area: three coordinate planes of the projected points (binary32,
 * nnz rounded up to 64) and the list of the fan's c_0 values.  Multiples of
 * 128 bytes. */
__host__ __device__ inline int td_fan_plane(int nnz) { return (nnz + 63) & ~63; }

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
    int off[8];         /* staged-layout offsets of the pivot rows [0, K-1) and of the other rows [4, 7) */
    int mode;           /* arithmetic of the projection (td_fan_project); -1: dependent tail */
    int stop;           /* early exit: some warp has reached 0 */
    int next;           /* the team's next fan in the tile */
    unsigned mx;        /* bit pattern of the largest |Y| */
    int cnt[8][4];      /* per warp of the team: c_0 values to sweep by pivot coordinate, dependent ones last */
    float sum[8][3];    /* per warp of the team: sums of |Y| by coordinate */
};

struct TdFan {
    float *y;           /* planes y, y + ny, y + 2 ny */
    uint16_t *list;
    TdFanHead *h;
    uint32_t *tab;      /* the team's histogram storage (strip tables, then a part per warp) */
    int T, tw, bar;     /* team size, this warp in the team, named barrier */
    int nt;             /* teams of the CTA */
    int ny;
};

__device__ __forceinline__ void td_team_sync(const TdFan &F)
{
    if (F.T == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(F.bar), "r"(F.T * 32) : "memory");
}

/* Position of point i in the planes: full blocks of 64 points interleave
 * points l and l + 32 (one 64-bit word a lane), the last partial block is in
 * order. */
__device__ __forceinline__ int td_fan_pos(int i, int nfull)
{
    return i < nfull ? (i & ~63) + 2 * (i & 31) + ((i >> 5) & 1) : i;
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
__device__ __forceinline__ void td_fan_tail(const float *xs, int npc, const int (&c)[D > 2 ? D - 2 : 1], int rowset,
                                            float mxall, TdFanHead *h, int lane)
{
    constexpr int KT = D - 3;
    if (lane == 0) h->mx = 0u;
    if constexpr (KT == 0) {
        if (lane < 3) h->off[4 + lane] = td_xidx(npc, 0, lane);
        if (lane == 0) {
            h->kappa = 1;
            h->mode = 0;
        }
    } else {
        auto minor = [&](const int (&r)[KT]) -> int64_t {
            int64_t m[KT][KT];
#pragma unroll
            for (int a = 0; a < KT; ++a)
#pragma unroll
                for (int b = 0; b < KT; ++b) m[a][b] = td_f2i(xs[td_xidx(npc, c[b + 1], r[a])]);
            return td_detk<KT>(m);
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
            h->d[ri][j] = minor(rr);
        }
        if (lane == 0) {
            h->kappa = kappa;
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
__device__ __forceinline__ void td_fan_project_m(const float *xs, int npc, int nnz, const TdFan &F, int lane)
{
    constexpr int KT = D - 3;
    const TdFanHead *h = F.h;
    const int nfull = nnz & ~63, npairs = ((nnz + 63) & ~63) >> 1;
    int op[KT > 0 ? KT : 1], oo[3];
    int64_t kap = 1, dd[3][KT > 0 ? KT : 1];
#pragma unroll
    for (int j = 0; j < KT; ++j) op[j] = h->off[j];
#pragma unroll
    for (int r = 0; r < 3; ++r) oo[r] = h->off[4 + r];
    if constexpr (KT > 0) {
        kap = h->kappa;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < KT; ++j) dd[r][j] = h->d[r][j];
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
                float a = (float)(int32_t)kap * xo[r].x, b = (float)(int32_t)kap * xo[r].y;
#pragma unroll
                for (int t = 0; t < KT; ++t) {
                    const float c = (float)(int32_t)dd[r][t];
                    a = fmaf(-c, xp[t].x, a);
                    b = fmaf(-c, xp[t].y, b);
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
        const int i = 2 * j0 + lane; /* points i and i + 32 */
        if (2 * j0 < nfull) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
                *reinterpret_cast<float2 *>(F.y + r * F.ny + 2 * j) = make_float2(yv[r][0], yv[r][1]);
        } else {
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                F.y[r * F.ny + i] = yv[r][0];
                F.y[r * F.ny + i + 32] = yv[r][1];
            }
        }
    }
    mx = __reduce_max_sync(TD_FULL, mx);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum[r] += __shfl_xor_sync(TD_FULL, sum[r], o);
    if (lane == 0) {
        atomicMax(&F.h->mx, mx);
#pragma unroll
        for (int r = 0; r < 3; ++r) F.h->sum[F.tw][r] = sum[r];
    }
}

/* Point at position pos of the planes (inverse of td_fan_pos). */
__device__ __forceinline__ int td_fan_point(int pos, int nfull)
{
    return pos < nfull ? (pos & ~63) + ((pos & 1) << 5) + ((pos & 63) >> 1) : pos;
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

template <int KC, int NB>
__device__ __forceinline__ uint32_t td_fan_strips(int nnz, const TdFan &F, int lo, int hi, int K, const float2 *dirs,
                                                  int best, int lane)
{
    constexpr int WORDS = TD_STRIP_WORDS(NB), LB = NB == 256 ? 8 : 7;
    static_assert(NB == 256 || NB == 128, "bins");
    constexpr unsigned MB = ((unsigned)(127 + 24 - LB) << 23) | 0x400000u; /* M = 1.5 * 2^(24 - LB): spacing 2 / NB */
    const float M = __uint_as_float(MB);
    const int T = F.T, st = TD_STRIP_MAX / K; /* dirs holds TD_STRIP_MAX + 1 directions */
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    for (int w = 0; w < T; ++w) {
        s0 += F.h->sum[w][0];
        s1 += F.h->sum[w][1];
        s2 += F.h->sum[w][2];
    }
    /* scales; a coordinate that vanishes throughout leaves no usable ratio */
    const float g0 = s0 > 0.f ? s2 * td_rcp(s0) : 0.f, g1 = s1 > 0.f ? s2 * td_rcp(s1) : 0.f;
    auto ratios = [&](int pos, float &A, float &B, float &h) -> bool {
        const float y0 = F.y[pos], y1 = F.y[pos + F.ny];
        h = F.y[pos + 2 * F.ny];
        const float r = td_rcp(h);
        A = y0 * (g0 * r);
        B = y1 * (g1 * r);
        const bool ok = h != 0.f && fabsf(A) + fabsf(B) <= 2048.f; /* false for NaN */
        if (!ok) A = B = 0.f;
        return ok;
    };
    /* byte address of a key's bin in the first strip's table, less 4 key */
    const unsigned tb = td_saddr(F.tab) + 16u + 4u * (NB / 2) - 4u * MB;
    uint32_t fail = 0u;
    const int b16 = min(best, 0x7fff);
    const uint32_t bias0 = (uint32_t)(0x8000 - b16) * 0x10001u;
    for (int k0 = 0; k0 < K; k0 += KC) {
        if (k0 > 0) td_team_sync(F); /* the previous tables are read */
        for (int j = 32 * F.tw + lane; j < KC * WORDS / 4; j += 32 * T)
            reinterpret_cast<uint4 *>(F.tab)[j] = make_uint4(0u, 0u, 0u, 0u);
        td_team_sync(F);
        const float2 *dk = dirs + k0 * st;
        for (int p0 = 32 * F.tw; p0 < nnz; p0 += 32 * T) {
            const int pos = p0 + lane; /* below ny: the planes are padded with zeros */
            float A, B, h;
            const uint32_t inc = ratios(pos, A, B, h) ? (h > 0.f ? 1u : 0x10000u) : 0u;
            int v = td_strip_key(A, B, dk[0], M);
            const float2 *d = dk;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int v2 = td_strip_key(A, B, *(d += st), M);
                td_reds_add(tb + 4u * (unsigned)max(v, v2) + 4u * WORDS * k, inc);
                td_reds_add(tb + 4u * (unsigned)min(v, v2) + 4u * (WORDS * k + NB), inc);
                v = v2;
            }
        }
        td_team_sync(F);
        /* prefix sums of both halves of every strip (packed counts of the two
         * signs, each below 2^12), the total after the second; the warps
         * share the arrays */
        for (int a = F.tw; a < 2 * KC; a += T) {
            constexpr int Q = NB / 128; /* quads per lane */
            uint32_t *t = F.tab + (a >> 1) * WORDS + 4 + (a & 1) * NB;
            uint4 q[Q];
            uint32_t sum = 0;
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                q[j] = reinterpret_cast<const uint4 *>(t)[Q * lane + j];
                q[j].x += sum;
                q[j].y += q[j].x;
                q[j].z += q[j].y;
                q[j].w += q[j].z;
                sum = q[j].w;
            }
            const uint32_t inc = (uint32_t)td_wscan_incl((int)sum, lane), ex = inc - sum;
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                q[j].x += ex;
                q[j].y += ex;
                q[j].z += ex;
                q[j].w += ex;
                reinterpret_cast<uint4 *>(t)[Q * lane + j] = q[j];
            }
            if ((a & 1) && lane == 31) t[NB] = inc;
        }
        td_team_sync(F);
        /* every strip's total is that of the counted points, by sign */
        const uint32_t bias = __byte_perm(F.tab[4 + 2 * NB], 0u, 0x1032) + bias0;
        int it = 0;
        for (int p0 = 32 * F.tw; p0 < nnz; p0 += 32 * T, ++it) {
            if ((p0 & ~63) >= hi || (p0 & ~63) + 64 <= lo) continue; /* no value of c_0 in this block */
            const int pos = p0 + lane;
            float A, B, h;
            uint32_t acc = ratios(pos, A, B, h) ? 0x80008000u : 0u;
            int v = td_strip_key(A, B, dk[0], M);
            const float2 *d = dk;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int v2 = td_strip_key(A, B, *(d += st), M);
                const uint32_t f = td_lds32(tb + 4u * (unsigned)min(v, v2) + 4u * (WORDS * k - 2));
                const uint32_t g = td_lds32(tb + 4u * (unsigned)max(v, v2) + 4u * (WORDS * k + NB + 1));
                /* low half: below and + with above and -; high half: the
                 * others; bit 15 of a half says that it reaches best */
                acc &= f - __byte_perm(g, 0u, 0x1032) + bias;
                v = v2;
            }
            if (acc != 0x80008000u) fail |= 1u << it;
        }
    }
    return fail;
}

/* Subsets to sweep one by one: the c_0 values lo <= i < hi whose bit is set in
 * the lanes' flags (bit it of a lane: position 32 (tw + T it) + lane), and the
 * dependent ones (Y = 0), counted by pivot coordinate. */
__device__ __forceinline__ void td_fan_count(int nnz, const TdFan &F, int lo, int hi, uint32_t fail, int lane)
{
    const int nfull = nnz & ~63;
    int cnt[4] = { 0, 0, 0, 0 };
    int it = 0;
    for (int p0 = 32 * F.tw; p0 < nnz; p0 += 32 * F.T, ++it) {
        if ((p0 & ~63) >= hi || (p0 & ~63) + 64 <= lo) continue;
        const int pos = p0 + lane, i = td_fan_point(pos, nfull);
        const float a0 = fabsf(F.y[pos]), a1 = fabsf(F.y[pos + F.ny]), a2 = fabsf(F.y[pos + 2 * F.ny]);
        const int k = a0 >= a1 ? (a0 >= a2 ? 0 : 2) : (a1 >= a2 ? 1 : 2);
        const bool in = i >= lo && i < hi, zero = fmaxf(a0, fmaxf(a1, a2)) == 0.f;
        const bool go = in && !zero && ((fail >> it) & 1u);
        cnt[3] += __popc(__ballot_sync(TD_FULL, in && zero));
        if (__any_sync(TD_FULL, go)) {
#pragma unroll
            for (int q = 0; q < 3; ++q) cnt[q] += __popc(__ballot_sync(TD_FULL, go && k == q));
        }
    }
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) F.h->cnt[F.tw][q] = cnt[q];
    }
}

/* The list of those subsets: c_0 values of pivot 0, 1, 2 in whole quads each,
 * then the at most three left over of each pivot, in the same order; n_k the
 * counts. */
__device__ __forceinline__ void td_fan_list(int nnz, const TdFan &F, int lo, int hi, uint32_t fail, int lane,
                                            const int (&nk)[3])
{
    const int nfull = nnz & ~63;
    const unsigned below = (1u << lane) - 1u;
    const int f0 = nk[0] & ~3, f1 = nk[1] & ~3, f2 = nk[2] & ~3;
    const int full[3] = { f0, f1, f2 }, base[3] = { 0, f0, f0 + f1 };
    const int left[3] = { f0 + f1 + f2, f0 + f1 + f2 + (nk[0] & 3), f0 + f1 + f2 + (nk[0] & 3) + (nk[1] & 3) };
    int run[3] = { 0, 0, 0 };
    for (int w = 0; w < F.tw; ++w)
#pragma unroll
        for (int q = 0; q < 3; ++q) run[q] += F.h->cnt[w][q];
    int it = 0;
    for (int p0 = 32 * F.tw; p0 < nnz; p0 += 32 * F.T, ++it) {
        if ((p0 & ~63) >= hi || (p0 & ~63) + 64 <= lo) continue;
        const int pos = p0 + lane, i = td_fan_point(pos, nfull);
        const float a0 = fabsf(F.y[pos]), a1 = fabsf(F.y[pos + F.ny]), a2 = fabsf(F.y[pos + 2 * F.ny]);
        const int k = a0 >= a1 ? (a0 >= a2 ? 0 : 2) : (a1 >= a2 ? 1 : 2);
        const bool in = i >= lo && i < hi && fmaxf(a0, fmaxf(a1, a2)) != 0.f && ((fail >> it) & 1u);
        if (!__any_sync(TD_FULL, in)) continue;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const unsigned b = __ballot_sync(TD_FULL, in && k == q);
            if (in && k == q) {
                const int rk = run[q] + __popc(b & below);
                F.list[rk < full[q] ? base[q] + rk : left[q] + rk - full[q]] = (uint16_t)i;
            }
            run[q] += __popc(b);
        }
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

/* The events of four subsets, into the warp's four tables.  off: byte
 * offsets (from the planes' start) of the planes a, b, p of each subset (all
 * four equal unless MIX).  Full blocks of 64 points take a pair a lane and
 * subset; the last partial block, when it holds at most 48 points, is
 * spread over the four subsets instead: lanes 8 g .. 8 g + 7 place 16 points
 * of subset g a step. */
template <bool MIX>
__device__ __forceinline__ void td_fan_points(unsigned ybase, int nnz, int lane, const unsigned (&oa)[4],
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
    td_f2x ya = 0, yb = 0, yp = 0; /* the next block's points, loaded a block ahead */
    if (!MIX && a < ae) {
        ya = td_lds64(a + oa[0]);
        yb = td_lds64(a + ob[0]);
        yp = td_lds64(a + op[0]);
    }
    for (; a < ae; a += 256u) {
        if constexpr (MIX) {
            td_fan_pair<0>(td_lds64(a + oa[0]), td_lds64(a + ob[0]), td_lds64(a + op[0]), na[0], nb[0], C, tb);
            td_fan_pair<TD_FAN_TABLE>(td_lds64(a + oa[1]), td_lds64(a + ob[1]), td_lds64(a + op[1]), na[1], nb[1], C, tb);
            td_fan_pair<2 * TD_FAN_TABLE>(td_lds64(a + oa[2]), td_lds64(a + ob[2]), td_lds64(a + op[2]), na[2], nb[2], C, tb);
            td_fan_pair<3 * TD_FAN_TABLE>(td_lds64(a + oa[3]), td_lds64(a + ob[3]), td_lds64(a + op[3]), na[3], nb[3], C, tb);
        } else {
            const td_f2x va = ya, vb = yb, vp = yp;
            const unsigned an = a + 256u < ae ? a + 256u : a;
            ya = td_lds64(an + oa[0]);
            yb = td_lds64(an + ob[0]);
            yp = td_lds64(an + op[0]);
            td_fan_pair<0>(va, vb, vp, na[0], nb[0], C, tb);
            td_fan_pair<TD_FAN_TABLE>(va, vb, vp, na[1], nb[1], C, tb);
            td_fan_pair<2 * TD_FAN_TABLE>(va, vb, vp, na[2], nb[2], C, tb);
            td_fan_pair<3 * TD_FAN_TABLE>(va, vb, vp, na[3], nb[3], C, tb);
        }
    }
    if (rem > 0 && rem <= 48) {
        const int g = lane >> 3;
        td_f2x ng, mg;
        td_lds_coef(coef + 16u * (unsigned)g, ng, mg);
        unsigned ga = oa[0], gb = ob[0], gp = op[0];
        if constexpr (MIX) {
#pragma unroll
            for (int s = 1; s < 4; ++s)
                if (g == s) {
                    ga = oa[s];
                    gb = ob[s];
                    gp = op[s];
                }
        }
        const unsigned tg = tb + (unsigned)g * TD_FAN_TABLE;
        unsigned b = ybase + 4u * (unsigned)(nnz - rem) + 8u * (unsigned)(lane & 7);
        for (int k = 0; k < rem; k += 16, b += 64u)
            td_fan_pair<0>(td_lds64(b + ga), td_lds64(b + gb), td_lds64(b + gp), ng, mg, C, tg);
    }
}

/* Subsets list[4 g .. 4 g + 3] of the fan (c[1..K) its tail): bounds for all
 * four from one pass over the points and 256 angular rows each, then the
 * exact sweep of those that do not reach best. */
template <int D>
__device__ __forceinline__ void td_fan_quad(const float *xs, int npc, int nnz, const TdFan &F, int g, int ntot,
                                            const TdFanConst &C, const int (&c)[D - 2], unsigned char *wb, unsigned char *mb,
                                            char *scratch, int np, const TdQuery *Q, int32_t *qmin, int blog2, int lane,
                                            int &best, uint64_t &n_exact, unsigned long long *ws)
{
    /* lane s < 4: subset s of the quad (past the end: subset 0 again) */
    const int nv = min(4, ntot - 4 * g);
    const int s = lane & 3;
    const int i = F.list[4 * g + (s < nv ? s : 0)];
    const float *yi = F.y + td_fan_pos(i, nnz & ~63);
    const float v0 = yi[0], v1 = yi[F.ny], v2 = yi[2 * F.ny];
    const float a0 = fabsf(v0), a1 = fabsf(v1), a2 = fabsf(v2);
    const int k = a0 >= a1 ? (a0 >= a2 ? 0 : 2) : (a1 >= a2 ? 1 : 2);
    const float yp = k == 0 ? v0 : (k == 1 ? v1 : v2);
    const float ya = k == 0 ? v1 : (k == 1 ? v2 : v0);
    const float yb = k == 0 ? v2 : (k == 1 ? v0 : v1);
    const float r = -td_rcp(yp);
    float4 *co = reinterpret_cast<float4 *>(mb + 16 + 192); /* the basis block's packed columns */
    __syncwarp(); /* the coefficients and the tables of the previous quad are read */
    if (lane < 4) {
        const float na = ya * r, nb = yb * r;
        co[lane] = make_float4(na, na, nb, nb);
    }
    {
        uint4 *z4 = reinterpret_cast<uint4 *>(wb);
        for (int j = lane; j < (4 * TD_FAN_TABLE >> 4); j += 32) z4[j] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncwarp();
    const unsigned pl = 4u * (unsigned)F.ny;
    const unsigned ybase = td_saddr(F.y), tab = td_saddr(wb), coef = td_saddr(co);
    unsigned oa[4], ob[4], op[4];
    if (__all_sync(TD_FULL, k == __shfl_sync(TD_FULL, k, 0))) {
        op[0] = k == 0 ? 0u : (k == 1 ? pl : 2u * pl);
        oa[0] = k == 0 ? pl : (k == 1 ? 2u * pl : 0u);
        ob[0] = k == 0 ? 2u * pl : (k == 1 ? 0u : pl);
        td_fan_points<false>(ybase, nnz, lane, oa, ob, op, coef, C, tab);
    } else {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int kt = __shfl_sync(TD_FULL, k, t);
            op[t] = kt == 0 ? 0u : (kt == 1 ? pl : 2u * pl);
            oa[t] = kt == 0 ? pl : (kt == 1 ? 2u * pl : 0u);
            ob[t] = kt == 0 ? 2u * pl : (kt == 1 ? 0u : pl);
        }
        td_fan_points<true>(ybase, nnz, lane, oa, ob, op, coef, C, tab);
    }
    __syncwarp();
    /* Pass 1: lane l scans rows 8 l .. 8 l + 7 of each table.  In a row the
     * walk stays within [P - cm, P + cp]; over the certified points only,
     * min(w, nc - w) is a lower bound (see td_sweep_filtered). */
    int mylb = INT_MAX; /* lane t: the bound of subset t */
    bool low = false;
#pragma unroll 1
    for (int t = 0; t < nv; ++t) {
        const uint4 *h4 = reinterpret_cast<const uint4 *>(wb + t * TD_FAN_TABLE) + 2 * lane;
        const uint4 qa = h4[0], qb = h4[1];
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
        if (lb < best) {
            low = true;
            /* At a row boundary the certified points are on known sides: the
             * walk value there plus all others is a halfspace count, so it
             * is not below V(S), and best may take it */
            const int ub = td_wmin(min(A + ex + lob, nc - (A + ex + hib))) + nnz - nc;
            if (ub < best) {
                best = ub;
                if (lane == 0) atomicMin(qmin, ub);
            }
        } else {
            n_exact += (uint64_t)(nnz - nc);
        }
    }
    if (low) {
        TdWarpSmem W;
        const TdScratch scr = td_scratch_at(scratch, np);
        td_warp_smem(W, wb, mb, scr);
#pragma unroll 1
        for (int t = 0; t < nv; ++t) {
            if (__shfl_sync(TD_FULL, mylb, t) >= best) continue;
            const int it = __shfl_sync(TD_FULL, i, t);
            const int V = td_sweep_one<D>(xs, npc, nnz, it, c, W, scr, Q, blog2, lane, best, ws);
            if (V < best) {
                best = V;
                if (lane == 0) atomicMin(qmin, V);
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

/* The fans of subset positions [r0, r1) of a query that this team takes: the
 * tile's fans are numbered in order and taken from the counter *ticket (the
 * first ones: the team's own number).  xs: the staged points; wb, mb: this
 * warp's histogram storage and basis block. */
template <int D>
__device__ __forceinline__ void td_team_sweep(const float *xs, int npc, int nnz, uint64_t r0, uint64_t r1, int mine,
                                              int *ticket, const TdFan &F, TdFanPlan &P, unsigned char *wb,
                                              unsigned char *mb, char *scratch, int np, const float2 *dirs,
                                              const TdQuery *Q, int32_t *qmin, int early_exit, int blog2, int rowset,
                                              int lane, int &best, unsigned long long *ws)
{
    constexpr int K = D - 2;
    if (r0 >= r1) return;
    int c[K];
    td_unrank_colex<K>(r0, nnz, c);
    float mxall = 0.f;
#pragma unroll
    for (int r = 0; r < D; ++r) mxall = fmaxf(mxall, (float)Q->mx[r]); /* < 2^22: exact */
    uint64_t n_sweeps = 0, n_dep = 0, n_exact = 0; /* n_sweeps, n_dep: in the team's first warp */
    uint64_t early = 0, early_quads = 0;           /* subsets left out by the early exit, those of quads */
    int gbest = best;
    uint64_t r = r0;
    if (F.tw == 0 && lane == 0) F.h->stop = 0;
    td_team_sync(F);
    for (int fan = 0; r < r1; ++fan) {
        const int lo = c[0];
        const uint64_t room = K >= 2 ? (uint64_t)(c[K >= 2 ? 1 : 0] - lo) : r1 - r;
        const int hi = lo + (int)(room < r1 - r ? room : r1 - r);
        if (fan == mine) {
            const bool stop = early_exit && F.h->stop; /* written before the last barrier only */
            if (F.tw == 0) {
                if (!stop) td_fan_tail<D>(xs, npc, c, rowset, mxall, F.h, lane);
                if (lane == 0) F.h->next = F.nt + atomicAdd(ticket, 1);
            }
            best = min(best, gbest);
            gbest = *reinterpret_cast<volatile int32_t *>(qmin);
            td_team_sync(F);
            mine = F.h->next;
            const int mode = stop ? -2 : F.h->mode;
            if (mode >= 0) {
                if (mode == 0) td_fan_project_m<D, 0>(xs, npc, nnz, F, lane);
                else if (mode == 1) td_fan_project_m<D, 1>(xs, npc, nnz, F, lane);
                else td_fan_project_m<D, 2>(xs, npc, nnz, F, lane);
                td_team_sync(F);
                const int ks = td_fan_choose(P, nnz, hi - lo);
                uint32_t fail = 0xffffffffu;
                if (ks > 0)
                    fail = F.T == 1   ? td_fan_strips<4, 128>(nnz, F, lo, hi, ks, dirs, best, lane)
                           : F.T == 2 ? td_fan_strips<8, 128>(nnz, F, lo, hi, ks, dirs, best, lane)
                                      : td_fan_strips<8, 256>(nnz, F, lo, hi, ks, dirs, best, lane);
                td_fan_count(nnz, F, lo, hi, fail, lane);
                td_team_sync(F);
                int nk[3] = { 0, 0, 0 }, nd = 0;
                for (int w = 0; w < F.T; ++w) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) nk[q] += F.h->cnt[w][q];
                    nd += F.h->cnt[w][3];
                }
                const int ntot = nk[0] + nk[1] + nk[2];
                if (F.tw == 0) {
                    n_dep += (uint64_t)nd;
                    n_sweeps += (uint64_t)(hi - lo - nd);
                }
                if (ks > 0) td_fan_learn(P, nnz, hi - lo, ntot);
                if (ntot > 0) {
                    td_fan_list(nnz, F, lo, hi, fail, lane, nk);
                    TdFanConst C;
                    {
                        const float X = __uint_as_float(F.h->mx);
                        const float cw = 48.0f * TD_U * X, M1 = 98305.0f; /* 1.5 * 2^16 + 1 */
                        C.c = td_pk(cw, cw);
                        C.nc = td_pk(-cw, -cw);
                        C.km = td_pk(M1, M1);
                    }
                    td_team_sync(F);
                    for (int g = F.tw; 4 * g < ntot; g += F.T) {
                        /* the query's minimum, lowered by other warps: read
                         * one quad ahead of its use */
                        best = min(best, gbest);
                        gbest = *reinterpret_cast<volatile int32_t *>(qmin);
                        if (early_exit && best <= 0) {
                            /* V = 0 is the least value: nothing can lower it */
                            early_quads += (uint64_t)min(4, ntot - 4 * g);
                            continue;
                        }
                        td_fan_quad<D>(xs, npc, nnz, F, g, ntot, C, c, wb, mb, scratch, np, Q, qmin, blog2, lane, best,
                                       n_exact, ws);
                    }
                }
                if (early_exit && best <= 0 && lane == 0) F.h->stop = 1;
            } else if (F.tw == 0) {
                if (stop) early += (uint64_t)(hi - lo);
                else n_dep += (uint64_t)(hi - lo);
            }
            td_team_sync(F); /* the planes, the list, the tables and the head are rewritten next */
        }
        r += (uint64_t)(hi - lo);
        if (K >= 2 && r < r1) {
            c[0] = hi - 1;
            td_next_colex<K>(c);
        }
    }
    best = min(best, gbest);
    if (lane == 0) {
        /* a subset that a quad left out after all is no sweep; the exact
         * sweeps move their uncertain points from ws[2] to ws[3] themselves */
        ws[0] += n_sweeps - early_quads;
        ws[1] += n_dep;
        ws[2] += (n_sweeps - early_quads) * (uint64_t)nnz - n_exact;
        ws[3] += n_exact;
        ws[7] += early + early_quads;
    }
}
