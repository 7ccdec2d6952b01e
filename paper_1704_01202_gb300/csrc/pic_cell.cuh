// Building blocks of the per-cell hot path: one warp (or, for large cells, a
// block of four) owns one cell and runs, in order, the canonical random
// ordering of its particles, the cell moments (double-float sums), binary
// e-e and e-i collisions, Lotz impact ionization, EOS-clamped recombination
// and, on rad steps, subshell photoionization and K-vacancy decay (k_cell);
// the Boris push and the charge-conserving deposit of the cell's particles
// follow in a second kernel in the same canonical order (k_push).
// Particles are staged in shared memory in that order.
//
// Determinism: every random number is keyed by (slab seed, particle id,
// step, purpose) and every ordering comes from a sort on Philox keys, so
// the result of a cell does not depend on where its particles sit in memory
// or on which warp handles it.  Sums run lane-strided over the canonical
// order with a fixed reduction tree; the current goes to global memory as
// 64-bit fixed point, whose addition is associative.
#pragma once
#include "pic_dev.cuh"

namespace pic {

constexpr unsigned FULL = 0xffffffffu;
// fixed-point scale of J: 2^40 (|J| < 2^22 per node); the FP64 build keeps
// 2^48 (|J| < 2^14), eight more bits for its 1e-12 comparison
constexpr double JFIX = sizeof(real) == 8 ? 281474976710656.0 : 1099511627776.0;

struct NewE {            // an electron created in this cell this step
    real ux, uy, uz, w;
    int meta;            // ion (position in the canonical order) | kind << 16
};

struct CellArgs {
    real4 *e0, *e1;     // electrons (xi, eta, ux, uy), (uz, w, id_lo, id_hi)
    int *ekey;           // next cell of each electron slot (-1: gone)
    const int *cs_e;     // cell start of electrons [ncell + 1]
    real4 *i0, *i1;     // ions (xi, eta, ux, uy), (uz, zfrac, id, Z | nK << 8)
    int *ikey;
    const int *cs_i;
    int *cnt_e, *cnt_i;  // per-cell counts of the next sort
    int *append;         // electrons appended this step
    int cap_e;           // electron capacity
    int *slab_app;       // [slab] electrons appended this step (budgeted slabs)
    int *slab_err;       // [slab] ERR_CAPACITY once a slab went beyond its budget
    int ncell;           // total cells (all slabs)
    const int *cell_slab;
    const SlabDev *slabs;
    const unsigned *steps;
    SlabTally *tally;
    ph2 *photons;
    const real *fldE;   // [3][npts] ex ey ez
    const real *fldB;   // [3][npts] bx by bz
    int npts;
    unsigned long long *J;   // [3][npts] fixed point
    const Tables *tab;
    const EosTable *eos;
    int *err;
    int *work;           // work counter
    const int *list;     // cell list (NULL: all cells)
    const int *n_list;   // number of cells in the list (device)
    int *ovf_list, *ovf_count;   // cells too large for this pass
    int cap_ce, cap_ci, cap_new; // per-cell capacities (staging; created electrons)
    NewE *nw;            // created-electron scratch: cap_new entries per team of the launch
};

// warp reductions: a fixed tree, result broadcast from lane 0 so every lane
// holds the same bits
__device__ __forceinline__ real wsum_f(real v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    return __shfl_sync(FULL, v, 0);
}

// dd_add is symmetric (TwoSum is exact either way round), so the butterfly
// gives every lane the bits of the tree (lane l + lane l + 16, then + 8, ...)
__device__ __forceinline__ dd wsum_dd(dd v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dd t{__shfl_xor_sync(FULL, v.hi, o), __shfl_xor_sync(FULL, v.lo, o)};
        v = dd_add(v, t);
    }
    return v;
}

// Two or four sums at once over the same trees: each level halves the lanes
// a sum needs, so the other sums use them (four sums cost six levels of
// arithmetic instead of twenty).
__device__ __forceinline__ dd wswap_add(dd a, dd b, bool up, int o)
{
    const dd mine = up ? b : a, give = up ? a : b;
    dd t{__shfl_xor_sync(FULL, give.hi, o), __shfl_xor_sync(FULL, give.lo, o)};
    return dd_add(mine, t);
}

__device__ __forceinline__ dd wtail_add(dd v, int from)
{
    for (int o = from; o > 0; o >>= 1) {
        dd t{__shfl_xor_sync(FULL, v.hi, o), __shfl_xor_sync(FULL, v.lo, o)};
        v = dd_add(v, t);
    }
    return v;
}

__device__ __forceinline__ dd wlane_dd(dd v, int src)
{
    return dd{__shfl_sync(FULL, v.hi, src), __shfl_sync(FULL, v.lo, src)};
}

__device__ __forceinline__ void wsum_dd2(dd &a, dd &b, int lane)
{
    const dd v = wtail_add(wswap_add(a, b, lane & 16, 16), 8);
    a = wlane_dd(v, 0);
    b = wlane_dd(v, 16);
}

__device__ __forceinline__ void wsum_dd4(dd &a, dd &b, dd &c, dd &d, int lane)
{
    const dd p = wswap_add(a, b, lane & 16, 16), q = wswap_add(c, d, lane & 16, 16);
    const dd v = wtail_add(wswap_add(p, q, lane & 8, 8), 4);
    a = wlane_dd(v, 0);
    b = wlane_dd(v, 16);
    c = wlane_dd(v, 8);
    d = wlane_dd(v, 24);
}

__device__ __forceinline__ int wsum_i(int v) { return __reduce_add_sync(FULL, v); }

// inclusive prefix over the lanes (fixed order)
__device__ __forceinline__ dd wscan_dd(dd v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        dd t{__shfl_up_sync(FULL, v.hi, o), __shfl_up_sync(FULL, v.lo, o)};
        if (lane >= o) v = dd_add(v, t);
    }
    return v;
}

// ---------------------------------------------------------------------
// canonical order inside a cell: ascending (64-bit Philox key, id)
// ---------------------------------------------------------------------
// The sort moves 32-bit words: the key's top 32 - SB bits over the entry's
// index (SB bits).  A compare-exchange is then one shuffle and one min or
// max, against two shuffles and a 64-bit compare for (48 key bits | index)
// words.  Entries whose words share all their key bits (n^2 2^SB / 2^33 pairs
// are expected in a cell of n: 2e-4 for 128 entries of one warp; by a team 0.48
// for 1000, so a pair in 0.38 of such cells, and 1.9 for 2000, in 0.85 of them)
// are put in (key, id) order afterwards, each run of
// them by the thread that finds its start, so the result is the full
// (key, id) order whatever SB is.

// keys and ids of a cell's records: Philox draws of the ids
struct RecKeys {
    const real4 *p1;         // second record words of the cell's first particle
    bool elec;
    unsigned long long seed;
    unsigned step;
    __device__ __forceinline__ unsigned long long id(int k) const
    {
        return elec ? rec_eid(p1[k]) : (unsigned long long)rec_iid(p1[k]);
    }
    __device__ __forceinline__ unsigned long long full(unsigned long long i) const
    {
        const U4 r = draw(seed, i, step, elec ? PU_PAIR_E : PU_PAIR_I);
        return ((unsigned long long)r.x << 32) | r.y;
    }
    __device__ __forceinline__ unsigned long long key(int k) const { return full(id(k)); }
    __device__ __forceinline__ unsigned top(int k) const
    {
        return draw(seed, id(k), step, elec ? PU_PAIR_E : PU_PAIR_I).x;
    }
};
// given keys and ids (the check entry)
struct GivenKeys {
    const unsigned long long *k_, *id_;
    __device__ __forceinline__ unsigned long long id(int k) const { return id_[k]; }
    __device__ __forceinline__ unsigned long long key(int k) const { return k_[k]; }
    __device__ __forceinline__ unsigned top(int k) const { return (unsigned)(k_[k] >> 32); }
};

// ascending bitonic sort of 32 E words of one warp, entry lane * E + j in
// v[j]; rolled over the sizes above E so that its code stays small
template <int E>
__device__ __forceinline__ void sort_words(unsigned (&v)[E], int lane)
{
#pragma unroll
    for (int size = 2; size <= E; size <<= 1) {
#pragma unroll
        for (int st = size >> 1; st > 0; st >>= 1) {
#pragma unroll
            for (int j = 0; j < E; ++j) {
                if (j & st) continue;
                // the last in-lane size alternates its direction by lane
                const bool asc = size < E ? (j & size) == 0 : (lane & 1) == 0;
                const unsigned lo = min(v[j], v[j | st]), hi = max(v[j], v[j | st]);
                v[j] = asc ? lo : hi;
                v[j | st] = asc ? hi : lo;
            }
        }
    }
#pragma unroll 1
    for (int ls = 2; ls <= 32; ls <<= 1) {           // size = ls * E
        const bool asc = (lane & ls) == 0;           // ls = 32: always
#pragma unroll 1
        for (int lm = ls >> 1; lm > 0; lm >>= 1) {
            const bool keep_min = ((lane & lm) == 0) == asc;
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const unsigned o = __shfl_xor_sync(FULL, v[j], lm);
                v[j] = keep_min ? min(o, v[j]) : max(o, v[j]);
            }
        }
#pragma unroll
        for (int st = E >> 1; st > 0; st >>= 1) {
#pragma unroll
            for (int j = 0; j < E; ++j) {
                if (j & st) continue;
                const unsigned lo = min(v[j], v[j | st]), hi = max(v[j], v[j | st]);
                v[j] = asc ? lo : hi;
                v[j | st] = asc ? hi : lo;
            }
        }
    }
}

// Runs of entries whose words share their key bits into (key, id) order:
// insertion within the run by the thread (of nt) at its start.  Permuting
// a run leaves its words' key bits in place, so the other threads' run
// boundaries do not move.
template <class Keys>
__device__ __noinline__ void order_ties(Keys K, unsigned *w, int n, int sb, int t, int nt)
{
    const unsigned mask = (1u << sb) - 1u;
    for (int k = t; k + 1 < n; k += nt) {
        const unsigned p = w[k] >> sb;
        if ((w[k + 1] >> sb) != p || (k > 0 && (w[k - 1] >> sb) == p)) continue;
        for (int q = k + 1; q < n && (w[q] >> sb) == p; ++q) {
            const unsigned x = w[q];
            const unsigned long long kx = K.key((int)(x & mask)), ix = K.id((int)(x & mask));
            int j = q - 1;
            while (j >= k) {
                const int y = (int)(w[j] & mask);
                const unsigned long long ky = K.key(y);
                if (!(ky > kx || (ky == kx && K.id(y) > ix))) break;
                w[j + 1] = w[j];
                --j;
            }
            w[j + 1] = x;
        }
    }
}

// one warp: w[k] = (key bits | index) of the entry at canonical position k
// of n <= 32 E entries.  Out of line: one copy serves both species.
template <int E, class Keys>
__device__ __noinline__ void order_warp(Keys K, unsigned *w, int n, int lane)
{
    constexpr int SB = E == 1 ? 5 : E == 2 ? 6 : E == 4 ? 7 : E == 8 ? 8 : 9;
    constexpr unsigned mask = (1u << SB) - 1u;
    unsigned v[E];
    // padding sorts last: an entry's word equals it only as entry 32 E - 1,
    // and then there is no padding
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int k = j * 32 + lane;
        v[j] = k < n ? (K.top(k) & ~mask) | (unsigned)k : ~0u;
    }
    sort_words<E>(v, lane);
    bool tie = false;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int k = lane * E + j;
        const unsigned nx = j + 1 < E ? v[j + 1 < E ? j + 1 : 0] : __shfl_down_sync(FULL, v[0], 1);
        tie |= k + 1 < n && (v[j] >> SB) == (nx >> SB);
        if (k < n) w[k] = v[j];
    }
    __syncwarp();
    if (__any_sync(FULL, tie)) {
        order_ties(K, w, n, SB, lane, 32);
        __syncwarp();
    }
}

// A team of TW warps (the whole block): each warp sorts a share of 32 E
// entries in registers, then every entry finds its place by its rank in the
// other shares (binary searches in shared memory).  w: n words out; buf:
// n words of scratch.
constexpr int TEAM_SB = 12;              // up to 4096 entries
template <int E, int TW, class Keys>
__device__ __noinline__ void order_team(Keys K, unsigned *w, unsigned *buf, int n, int warp, int lane)
{
    constexpr unsigned mask = (1u << TEAM_SB) - 1u;
    unsigned v[E];
    const int base = warp * 32 * E;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int k = base + j * 32 + lane;
        v[j] = k < n ? (K.top(k) & ~mask) | (unsigned)k : ~0u;
    }
    sort_words<E>(v, lane);
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int k = base + lane * E + j;
        if (k < n) buf[k] = v[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < E; ++j) {
        if (base + lane * E + j >= n) continue;
        int rank = lane * E + j;
        for (int o = 0; o < TW; ++o) {
            if (o == warp) continue;
            int lo = o * 32 * E, hi = min(n, lo + 32 * E);   // first word above v[j]
            const int b = lo;
            while (lo < hi) {
                const int md = (lo + hi) >> 1;
                if (buf[md] < v[j]) lo = md + 1; else hi = md;
            }
            rank += max(lo - b, 0);
        }
        w[rank] = v[j];
    }
    __syncthreads();
    bool tie = false;
    for (int k = warp * 32 + lane; k + 1 < n; k += 32 * TW) tie |= (w[k] >> TEAM_SB) == (w[k + 1] >> TEAM_SB);
    if (__syncthreads_or(tie)) {
        order_ties(K, w, n, TEAM_SB, warp * 32 + lane, 32 * TW);
        __syncthreads();
    }
}

// the canonical order of a cell of n entries by a team of TW warps: w[k] &
// (return value) is the index of the entry at position k (buf: a team's
// scratch, n words)
template <int RMAX, int TW, class Keys>
__device__ __forceinline__ unsigned order_cell(const Keys &K, unsigned *w, unsigned *buf, int n, int warp, int lane)
{
    if constexpr (TW == 1) {
        if (n <= 32) { order_warp<1>(K, w, n, lane); return 31u; }
        if (n <= 64) { order_warp<2>(K, w, n, lane); return 63u; }
        if (RMAX <= 128 || n <= 128) { order_warp<4>(K, w, n, lane); return 127u; }
        if constexpr (RMAX > 128) {
            if (n <= 256) { order_warp<8>(K, w, n, lane); return 255u; }
            order_warp<16>(K, w, n, lane);
        }
        return 511u;
    } else {
        if (n <= 32 * TW) order_team<1, TW>(K, w, buf, n, warp, lane);
        else if (n <= 64 * TW) order_team<2, TW>(K, w, buf, n, warp, lane);
        else if (n <= 128 * TW) order_team<4, TW>(K, w, buf, n, warp, lane);
        else if (n <= 256 * TW) order_team<8, TW>(K, w, buf, n, warp, lane);
        else order_team<16, TW>(K, w, buf, n, warp, lane);
        return (1u << TEAM_SB) - 1u;
    }
}

__device__ __forceinline__ real cic_w(real x, int node)
{
    real d = r_fabs(x - (real)node);
    return d < RF(1.0) ? RF(1.0) - d : RF(0.0);
}

// Shared-memory staging of one cell, by the team (one warp, or the whole
// block) that owns it.  Every array is in the cell's canonical order: a
// warp's lanes read neighbouring entries, without bank conflicts and
// without an index to load first.
struct CellMem {
    real4 *eu;                 // [cap_ce] ux uy uz w
    real2 *epos;               // [cap_ce] positions in the cell
    unsigned long long *eid;    // [cap_ce]
    real2 *ew;                 // [max(cap_ce, cap_ci)] scratch: sort words; kinetic energy and w beta of each
                                //   electron; weight taken by recombination
    real4 *rn;                 // [cap_ce] e-i collisions' draws (launches of small cells, coll_draws_staged)
    real4 *iu;                 // [cap_ci] ux uy uz zfrac
    real2 *ipos;               // [cap_ci]
    int *ist;                   // [cap_ci] Z | nK << 8
    unsigned int *iid;          // [cap_ci]
    int *nrec;                  // [cap_ci] recombinations of each ion
    NewE *nw;                   // [cap_new] in global memory: the team's slice of the scratch
    real *dE;                  // [16] continuum lowering per charge state
    real *Pz;                  // [16] impact-ionization probability per charge
    real4 *lz;                 // [TW][LOTZ_SETS][NS] Lotz constants of a charge state (a warp's four sets): P, 1/P, ln P, a q
    dd *ph;                     // [2 MAXB] photon bin scratch
    int *phc;                   // [MAXB] events per bin so far
    dd *bc;                     // [8] sums a warp hands to its team
};

constexpr int LOTZ_SETS = 4;     // a warp

// shared-memory pieces start on 16 B (FP32) or 32 B (FP64: real4 is 32 B)
constexpr size_t kSmAlign = sizeof(real4) > 16 ? 32 : 16;
__host__ __device__ inline size_t amem(size_t x) { return (x + kSmAlign - 1) & ~(kSmAlign - 1); }

// The launches that stage at most 128 entries, a warp a cell, form the draws of the e-i
// collisions before the chains of collisions (see there): 16 bytes more an
// electron, which would cost the larger ones resident warps.
__host__ __device__ constexpr bool coll_draws_staged(int ce, int ci, int tw) { return ce <= 128 && ci <= 128 && tw == 1; }

// Shared memory of a team of tw warps staging up to ce electrons and ci ions.  The
// electrons a cell creates in a step (up to 3 per ion: impact, photo- and
// Auger ionization) are rare; they live in the team's slice of a global
// scratch, which keeps the staging of large cells small.
__host__ __device__ inline size_t cell_mem_bytes(int ce, int ci, int tw)
{
    const int cm = ce > ci ? ce : ci;
    return amem((size_t)ce * sizeof(real4)) + amem((size_t)ce * sizeof(real2)) + amem((size_t)ce * 8) +
           amem((size_t)cm * sizeof(real2)) + (coll_draws_staged(ce, ci, tw) ? amem((size_t)ce * sizeof(real4)) : 0) +
           amem((size_t)ci * sizeof(real4)) + amem((size_t)ci * sizeof(real2)) +
           3 * amem((size_t)ci * 4) + 2 * amem(16 * sizeof(real)) + amem(tw * LOTZ_SETS * NS * sizeof(real4)) +
           amem(2 * MAXB * sizeof(dd)) + amem(MAXB * 4) + amem(8 * sizeof(dd));
}

__device__ inline CellMem carve(char *base, int ce, int ci, int tw, NewE *nw)
{
    CellMem m;
    const int cm = ce > ci ? ce : ci;
    char *p = base;
    m.eu = (real4 *)p; p += amem((size_t)ce * sizeof(real4));
    m.epos = (real2 *)p; p += amem((size_t)ce * sizeof(real2));
    m.eid = (unsigned long long *)p; p += amem((size_t)ce * 8);
    m.ew = (real2 *)p; p += amem((size_t)cm * sizeof(real2));
    m.rn = (real4 *)p;
    if (coll_draws_staged(ce, ci, tw)) p += amem((size_t)ce * sizeof(real4));
    m.iu = (real4 *)p; p += amem((size_t)ci * sizeof(real4));
    m.ipos = (real2 *)p; p += amem((size_t)ci * sizeof(real2));
    m.ist = (int *)p; p += amem((size_t)ci * 4);
    m.iid = (unsigned int *)p; p += amem((size_t)ci * 4);
    m.nrec = (int *)p; p += amem((size_t)ci * 4);
    m.nw = nw;
    m.dE = (real *)p; p += amem(16 * sizeof(real));
    m.Pz = (real *)p; p += amem(16 * sizeof(real));
    m.lz = (real4 *)p; p += amem(tw * LOTZ_SETS * NS * sizeof(real4));
    m.ph = (dd *)p; p += amem(2 * MAXB * sizeof(dd));
    m.phc = (int *)p; p += amem(MAXB * 4);
    m.bc = (dd *)p;
    return m;
}

// grid of one slab, as the deposit of long moves takes it
struct SlabGrid {
    int nx, ny, W;       // W = nx + 1 points per row
    int npts;            // stride between components
    int fo;              // first grid point of the slab
};

// ---------------------------------------------------------------------
// current deposit
// ---------------------------------------------------------------------
struct JAcc2 { real x[3][4], y[4][3], z[4][4]; };
struct JAcc1 { real x[3], y[4], z[4]; };

// v * 2^40 rounded to a 64-bit integer with FP32 and integer instructions
// only (|v| < 2^22): the high part is split off exactly at 2^31 (the
// FP64 build rounds v * JFIX directly)
__device__ __forceinline__ long long fix40(real v)
{
#ifdef PIC_FP64
    return __double2ll_rn(v * JFIX);
#else
    float x = v * 1099511627776.0f;                     // exact: power-of-two scale
    float qh = truncf(x * 4.656612873077393e-10f);      // x / 2^31, integer part
    float r = fmaf(-qh, 2147483648.0f, x);               // exact remainder, |r| < 2^31
    long long lo = (long long)__float2int_rn(fminf(fmaxf(r, -2147483520.0f), 2147483520.0f));
    return ((long long)(int)qh << 31) + lo;
#endif
}

__device__ __forceinline__ void jatomic(unsigned long long *J, real v)
{
    if (v != RF(0.0)) atomicAdd(J, (unsigned long long)fix40(v));
}

// Esirkepov weights of one sub-cell move, stencil anchored at cell (ax, ay)
// offsets -1..2; start (x0, y0), end (x1, y1) relative to the anchor cell
__device__ __forceinline__ void esirkepov2(real x0, real y0, real x1, real y1, real qw, real qwbz,
                                           real frac, JAcc2 &A)
{
    real S0x[4], S1x[4], S0y[4], S1y[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        S0x[a] = cic_w(x0, a - 1); S1x[a] = cic_w(x1, a - 1);
        S0y[a] = cic_w(y0, a - 1); S1y[a] = cic_w(y1, a - 1);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        real acc = RF(0.0);
        real sy = S0y[b] + RF(0.5) * (S1y[b] - S0y[b]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc += (S1x[a] - S0x[a]) * sy;
            A.x[a][b] -= qw * acc;
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        real acc = RF(0.0);
        real dsx = S1x[a] - S0x[a];
        real sx = S0x[a] + RF(0.5) * dsx;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            acc += (S1y[b] - S0y[b]) * sx;
            A.y[a][b] -= qw * acc;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            real dsy = S1y[b] - S0y[b];
            real wz = S0x[a] * S0y[b] + RF(0.5) * dsx * S0y[b] + RF(0.5) * S0x[a] * dsy + dsx * dsy * (RF(1.0) / RF(3.0));
            A.z[a][b] += qwbz * wz * frac;
        }
    }
}

__device__ __forceinline__ void esirkepov1(real x0, real x1, real qw, real qwby, real qwbz, real frac, JAcc1 &A)
{
    real S0x[4], S1x[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) { S0x[a] = cic_w(x0, a - 1); S1x[a] = cic_w(x1, a - 1); }
    real acc = RF(0.0);
#pragma unroll
    for (int a = 0; a < 3; ++a) { acc += S1x[a] - S0x[a]; A.x[a] -= qw * acc; }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        real s = RF(0.5) * (S0x[a] + S1x[a]);
        A.y[a] += qwby * s * frac;
        A.z[a] += qwbz * s * frac;
    }
}

// a move of one cell or more: equal sub-cell segments, each deposited
// straight to global memory around its own start cell
__device__ __noinline__ void deposit_long(const SlabGrid &g, unsigned long long *J, int npts, int fo, int cx, int cy,
                             real x0, real y0, real x1, real y1, real qw, real qwby, real qwbz)
{
    real ax = r_fabs(x1 - x0), ay = g.ny > 1 ? r_fabs(y1 - y0) : RF(0.0);
    int nseg = (int)r_floor(r_fmax(ax, ay)) + 1;
    for (int k = 0; k < nseg; ++k) {
        real a0 = (real)k / nseg, a1 = (real)(k + 1) / nseg;
        real xa = x0 + a0 * (x1 - x0), xb = x0 + a1 * (x1 - x0);
        real ya = y0 + a0 * (y1 - y0), yb = y0 + a1 * (y1 - y0);
        int sx = (int)r_floor(xa), sy = g.ny > 1 ? (int)r_floor(ya) : 0;
        real f = RF(1.0) / nseg;
        if (g.ny == 1) {
            JAcc1 A = {};
            esirkepov1(xa - sx, xb - sx, qw, qwby, qwbz, f, A);
            for (int a = 0; a < 4; ++a) {
                int i = cx + sx - 1 + a;
                if (a < 3 && i >= 0 && i < g.nx) jatomic(J + fo + i, A.x[a]);
                if (i >= 0 && i <= g.nx) {
                    jatomic(J + npts + fo + i, A.y[a]);
                    jatomic(J + 2 * npts + fo + i, A.z[a]);
                }
            }
        } else {
            JAcc2 A = {};
            esirkepov2(xa - sx, ya - sy, xb - sx, yb - sy, qw, qwbz, f, A);
            for (int a = 0; a < 4; ++a) {
                int i = cx + sx - 1 + a;
                for (int b = 0; b < 4; ++b) {
                    int j = (cy + sy - 1 + b) % g.ny; if (j < 0) j += g.ny;
                    size_t o = (size_t)fo + (size_t)j * g.W + i;
                    if (a < 3 && i >= 0 && i < g.nx) jatomic(J + o, A.x[a][b]);
                    if (b < 3 && i >= 0 && i <= g.nx) jatomic(J + npts + o, A.y[a][b]);
                    if (i >= 0 && i <= g.nx) jatomic(J + 2 * npts + o, A.z[a][b]);
                }
            }
        }
    }
}

}  // namespace pic
