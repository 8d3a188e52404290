/*
 * td_internal.h -- structures shared by the host side and the kernels of
 * libtukeydepth.so (not part of the public ABI).
 */
#pragma once
#include <stdint.h>

#define TD_MAXD 6
#define TD_NDIM 5            /* effective dimensions 2..6 with a subset loop */
#define TD_TICKET_STRIDE 16  /* work counters 128 bytes apart */
#define TD_DIRECT_WIDE (-2)  /* TdQuery.direct of a query whose centred coordinates exceed the fast
                                kernels' limit: answered by the wide kernel (td_wide.cuh) */
#define TD_NOCT 12           /* octaves of the nonzero point count: ceil(log2 nnz) in [0, 11] */

/* octave of a row of nnz nonzero points (1 <= nnz <= 2048): ceil(log2 nnz) */
static inline __host__ __device__ int td_octave(int nnz)
{
    int b = 0;
    while (b < TD_NOCT - 1 && (1 << b) < nnz) ++b;
    return b;
}

/* Warps per CTA of the sweep kernel of effective dimension D.  D = 2: a warp
 * works alone, 32 an SM.  D >= 3: 16 warps an SM by their registers (up to 128 a
 * thread; 24 warps at 80 registers spill and were slower), fewer where the
 * shared memory of long rows does not allow them: at D = 4 one CTA of 8 beyond
 * 1792 points; at D = 5 three CTAs of 4 beyond 416 and two beyond 896, at D = 6
 * three beyond 416 and two beyond 640.  D = 3, 4: a fan of long rows is taken
 * by up to 8 warps (4-warp CTAs: W2 3.77 ms against 3.20).  D = 5, 6: fans are
 * short and warps take them alone, so that a CTA only needs to be large enough
 * to share its copy of the rows; 8-warp CTAs were no faster (W4 31.9 ms
 * against 31.4, p = 6 12.3 against 11.9: within what runs differ by). */
static inline __host__ __device__ constexpr int td_sweep_warps(int D) { return D == 3 || D == 4 ? 8 : 4; }

/* Tile sizes are given in subsets per warp for CTAs of this many warps. */
#define TD_TILE_WARPS 8

/* a / b for b > 0, by the 32-bit unsigned divide when both operands fit */
static inline __host__ __device__ int64_t td_div_nonneg(int64_t a, int64_t b)
{
    if ((((uint64_t)a | (uint64_t)b) >> 32) == 0) return (int64_t)((uint32_t)a / (uint32_t)b);
    return a / b;
}

/* Subsets per warp and tile for a query of effective dimension D and nnz
 * nonzero points, in a call of that many subset positions times points
 * (total, over all queries) on a GPU of sms SMs: 2^19 / nnz (a tile is 4096
 * subsets at 1000 points: a few fans a team, so that few are cut at a tile's
 * ends and the teams' wait for the slowest is short; half that size made W2
 * 3.54 ms 4.09), at most 2048, and so few that the call has tiles for four
 * rounds of the resident CTAs -- three at D = 3, where a tile is one fan and
 * a cut costs it a second pass over the points (four: 886 us for the 1000
 * rows of own_depths_p3, 795 with three) -- since some queries' exact steps
 * take far longer than others' and with one or two rounds the last tiles run
 * alone.  One tile for 1/608 of the work at every D, which at D = 5, 6 is a
 * single round: 2 queries of p = 5, n = 200 998 us a call, 574 so; 16 of p =
 * 6, n = 40 1084 and 878; 64 of p = 3, n = 1000 with coordinates -2 .. 2 5540
 * and 4460.  At least 2 (16 a tile: 4 made W1, 16 queries of 300 subsets, 113
 * us a call against 104, 1 made it 112). */
static inline __host__ __device__ int td_auto_spw(int D, int nnz, int64_t total, int sms)
{
    const int64_t n = nnz > 0 ? nnz : 1;
    const int64_t ctas = (int64_t)sms * (16 / td_sweep_warps(D));
    int64_t s = (1 << 19) / n;
    const int64_t cap = td_div_nonneg(total, (D == 3 ? 3 : 4) * ctas * TD_TILE_WARPS * n);
    s = s < cap ? s : cap;
    return s < 2 ? 2 : (s > 2048 ? 2048 : (int)s);
}

/* The same with a tuned size (0: none): it was found on a call of 64 tiles and
 * more a resident block, and where there are fewer than 24 its larger tiles
 * cost more at the end than they save (W2, 3.6 ms with tiles for 25 rounds:
 * 4.25 with tuned ones for 13), so there the rule's size or the one that makes
 * 24 rounds is taken, whichever is larger. */
static inline __host__ __device__ int td_tuned_spw(int D, int nnz, int64_t total, int sms, int tuned)
{
    const int rule = td_auto_spw(D, nnz, total, sms);
    if (tuned <= rule) return tuned > 0 ? tuned : rule;
    const int64_t n = nnz > 0 ? nnz : 1;
    const int64_t cap = td_div_nonneg(total, 24 * (int64_t)sms * (16 / td_sweep_warps(D)) * TD_TILE_WARPS * n);
    return cap >= tuned ? tuned : (cap > rule ? (int)cap : rule);
}

/* The middle of two keys given as bit patterns of positive binary32 values
 * (below 2^31 each: their sum needs all 32 bits, so it is unsigned). */
static inline __host__ __device__ int td_key_middle(int a, int b) { return (int)(((uint32_t)a + (uint32_t)b) >> 1); }

/* Blocks of a sweep kernel whose scratch holds `warps` warps in all: as many as
 * are resident, and no fewer warps where the dimension's blocks are narrow (80
 * blocks of any width: 322 us for 4096 queries of p = 2, n = 512 and 12.3 ms
 * for 64 of p = 6, n = 40 without allocation, 237 us and 6.9 ms by warps). */
static inline __host__ __device__ int td_capped_grid(int D, int sms, int occ, int warps)
{
    const int most = warps / td_sweep_warps(D), resident = sms * occ;
    return resident < most ? resident : most;
}

/* Largest |X_ij - z_j| (every coordinate) the fast kernels take for
 * dimension p: it keeps every exact intermediate in 64-bit (coordinates,
 * minors, projections) or 128-bit (cross products) integers, every
 * coordinate exact in binary32, and inside the window of the magic-constant
 * float-to-int conversion (|v| <= 2^22).  Queries beyond it go to the wide
 * kernel. */
static inline __host__ __device__ int64_t td_coord_limit_of(int p)
{
    switch (p) {
    case 1:
    case 2:
    case 3: return 4194303; /* 2^22 - 1 */
    case 4: return 524287;  /* 4 * 2 M^2 * M < 2^62 */
    case 5: return 16383;   /* 5 * 3^(3/2) M^3 * M < 2^62 */
    case 6: return 2047;    /* 6 * (2M)^4 * M < 2^62 */
    default: return 0;
    }
}

/* Per-query state written by the set-up kernel (one per query). */
struct TdQuery {
    int32_t set;           /* dataset index */
    int32_t n;             /* data points of the dataset */
    int32_t nnz;           /* centred points x_i = X_i - z that are nonzero */
    int32_t Z;             /* centred points equal to zero (counted by every closed halfspace) */
    int32_t d;             /* rank of the nonzero centred points (effective dimension) */
    int32_t k;             /* subset size d - 2 of Algorithm 1, or -1 when there is no subset loop */
    int32_t direct;        /* final count when there is no subset loop (nnz == 0 or d <= 1, or the
                              wide kernel's result), -1 when there is one, TD_DIRECT_WIDE while a
                              query beyond the fast kernels' limit waits for the wide kernel */
    int32_t amax;          /* max |x_ij| over every coordinate (saturated at INT32_MAX) */
    int32_t piv[TD_MAXD];  /* coordinates on which the span of the points projects injectively */
    int32_t mx[TD_MAXD];   /* max |x_i| per projected coordinate (FP32 error bounds) */
    int64_t nsub;          /* subset positions C(nnz, k) of the whole loop */
    int64_t lo, hi;        /* subset positions [lo, hi) handled by this call (shard) */
};

/* One dataset inside the device arenas. */
struct TdSet {
    int64_t x_off;  /* offset of X (n x p int32) in the data arena, in int32 elements */
    int32_t n, p;
    int32_t slice_index, slice_count; /* this call handles slice slice_index of slice_count contiguous
                                         ranges of each query's subset positions (the stream's time
                                         slices; slice_count <= 1: the call's shard) */
};

/* Statistics counters accumulated on the device. */
struct TdCounters {
    unsigned long long sweeps, dependent, filtered_points, exact_points, tight, resolved;
    unsigned long long errors;  /* device-side consistency failures (must stay 0) */
    unsigned long long early;   /* subsets not swept because their query had reached 0 (early exit) */
    unsigned long long adia_pops, adia_subsets, adia_union, adia_fallback; /* Algorithm 3 search */
    unsigned long long rescanned; /* sweeps whose bounds did not reach the minimum: the exact steps */
    unsigned long long wide;      /* queries the set-up flagged TD_DIRECT_WIDE */
    unsigned long long dims;      /* bit d: some query of effective dimension d has a subset loop */
    unsigned long long work;      /* subset positions times nonzero points, over the queries with k >= 1 */
};

/* Parameters of the work-queue launches. */
struct TdLaunch {
    const int32_t *X;        /* data arena */
    const int32_t *Zq;       /* query points, m_total x p_q (row stride TD_MAXD) */
    const TdSet *sets;
    TdQuery *q;              /* per query */
    const int32_t *qset;     /* dataset of every query (null: q[].set holds it already) */
    int32_t nq;              /* number of queries */
    int32_t warps;           /* warps per CTA */
    int32_t sms;             /* SMs of the GPU (or as many as the call's CTAs fill) */
    const int32_t *order;    /* work order of the queries (a permutation of [0, nq)) */
    int64_t *tile_prefix;    /* TD_NDIM x (nq + 1) prefix sums of tiles, per dimension, in work order */
    int32_t *tile_size;      /* subsets per tile, per query */
    unsigned long long *ticket;  /* work-queue counters, one per dimension (stride TD_TICKET_STRIDE) */
    int32_t *qmin;           /* per-query minimum of V(S) over the processed subsets */
    int32_t *out;            /* per-query output */
    TdCounters *ctr;
    int64_t shard_index, shard_count;
    int32_t spw;             /* subsets per warp per tile (0 = the tuned table, else by size) */
    uint16_t spw_tab[TD_NDIM][TD_NOCT]; /* tuned subsets per warp by dimension and octave (0 = by size) */
    int32_t blog2;           /* angular buckets log2 (0 = by size) */
    int32_t nmax;            /* largest nnz over the queries (smem sizing) */
    int32_t pmax;            /* largest p over the datasets */
    char *scratch;           /* per-warp global scratch for the exact tight-set path */
    int64_t scratch_per_warp;
    int32_t early_exit;      /* nonzero: seed qmin with the data-direction bound, stop a query at 0 */
    int32_t adia;            /* nonzero: Algorithm 3 (search kernel before the sweep) */
    int32_t critical;        /* nonzero: Proposition 1 with r = p-1 (subsets of d-1 points) */
    int32_t unseeded;        /* nonzero: qmin starts at +inf, not at the data-direction bound */
    uint16_t *perm;          /* Algorithm 3: staging position of every nonzero point, per query, or null */
    int64_t perm_stride;     /* entries per query in perm */
    uint64_t *adia_keys;     /* Algorithm 3 node tables, per CTA of the search kernel */
    int32_t *adia_dep;
    int32_t *adia_stack;
};
