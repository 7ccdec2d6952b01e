// Boris push and charge-conserving deposit, one warp, or a block of four,
// per cell.
//
// A cell's particles are visited in the canonical order, which is the order
// the collision kernel left them in.  Lane L takes canonical positions L,
// L+32, ...; each lane stores its stencil contributions in a shared-memory
// column, the rows of each batch are summed in a fixed order and added, batch
// by batch, to the running total of their node, and the cell's totals go to
// the global grid as 2^40 fixed point, whose addition is associative.  The
// current is therefore bit-reproducible, and the same for any team.
#pragma once
#include "pic_cell.cuh"

namespace pic {

struct PushArgs {
    real4 *e0, *e1;
    int *ekey;
    const int *cs_e;
    real4 *i0, *i1;
    int *ikey;
    const int *cs_i;
    int *cnt_e, *cnt_i;
    const int *append;        // electrons appended this step (after the sorted range)
    int cap_e;
    int ncell;
    const int *cell_slab;
    const SlabDev *slabs;
    SlabTally *tally;
    const real *fldE, *fldB;
    int npts;
    unsigned long long *J;
    int *err;
    int *work;
};


// Per-warp staging of the stencil contributions: row k (node), column lane.
// The row pitch of 36 words lets 16-byte row reads of 8 lanes and the
// column stores of a warp fall on different banks.
// (the FP64 build halves the warps per CTA: its rows are twice as wide)
constexpr int PUSH_TEAM = 4, PUSH_NEW_CTAS = 64;
constexpr int JROWS = 40, JPITCH = 36, PUSH_WARPS = sizeof(real) == 8 ? 4 : 8;
struct __align__(kSmAlign) JStage { real v[JROWS * JPITCH]; };
// jrows reads the rows as real4 (32-byte aligned in the FP64 build)
static_assert(alignof(JStage) >= alignof(real4) && JPITCH * sizeof(real) % alignof(real4) == 0 &&
                  sizeof(JStage) % alignof(real4) == 0,
              "alignment of the stencil rows");

__device__ __forceinline__ void jput(real *col, int k, real v) { col[k * JPITCH] = v; }

// Row sums of one batch: row k is summed as four interleaved partial sums
// in ascending order, then pairwise.  Rows below FULLROWS (a multiple of 32,
// or 0): a lane each, four words at a time, t[0].  The remaining rows: a lane
// per partial sum, eight rows at a time, t[1..], the same total in the four
// lanes of a row.  A row's sum has the same bits either way.
template <int NROWS>
__device__ __forceinline__ void jrows(const real *sj, int lane, real (&t)[3])
{
    constexpr int FULLROWS = NROWS / 32 * 32;
    __syncwarp();
    if constexpr (FULLROWS > 0) {
        const real4 *r = reinterpret_cast<const real4 *>(sj + lane * JPITCH);
        real4 s4 = r[0];
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            const real4 v = r[q];
            s4.x += v.x; s4.y += v.y; s4.z += v.z; s4.w += v.w;
        }
        t[0] = (s4.x + s4.y) + (s4.z + s4.w);
    }
#pragma unroll
    for (int g = 0; FULLROWS + 8 * g < NROWS; ++g) {
        const int k = FULLROWS + 8 * g + (lane >> 2);
        real v = RF(0.0);
        if (k < NROWS) {
            const real *r = sj + k * JPITCH + (lane & 3);
            v = r[0];
#pragma unroll
            for (int q = 1; q < 8; ++q) v += r[4 * q];
        }
        v += __shfl_xor_sync(FULL, v, 1);
        v += __shfl_xor_sync(FULL, v, 2);
        t[1 + g] = v;
    }
    __syncwarp();
}

// Linear weights at the stencil nodes -1..2 of a start point in [0, 1): only
// the nodes 0 and 1 are not zero (1 - |x - 1| as 1 - (1 - x)).
struct Start { real w1, w2; };
__device__ __forceinline__ Start start_w(real x)
{
    const real d = RF(1.0) - x;
    return Start{d, RF(1.0) - d};
}

// 2D Esirkepov weights of one sub-cell move (offsets relative to the cell,
// stencil nodes -1..2); order of the rows: jx[a][b] (12), jy[a][b] (12),
// jz[a][b] (16).  The fused products are written out: the current's last
// bits decide where a sort puts a particle later.
__device__ __forceinline__ void esirkepov2_w(real x0, real y0, real x1, real y1, real qw, real qwbz,
                                             real *col)
{
    const Start sx0 = start_w(x0), sy0 = start_w(y0);
    const real S0x[4] = {RF(0.0), sx0.w1, sx0.w2, RF(0.0)}, S0y[4] = {RF(0.0), sy0.w1, sy0.w2, RF(0.0)};
    real dx[4], dy[4], sx[4], sy[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const bool z = a == 0 || a == 3;            // S0 = 0
        const real S1x = cic_w(x1, a - 1), S1y = cic_w(y1, a - 1);
        dx[a] = z ? S1x : S1x - S0x[a];
        dy[a] = z ? S1y : S1y - S0y[a];
        sx[a] = z ? RF(0.5) * dx[a] : r_fma(RF(0.5), dx[a], S0x[a]);
        sy[a] = z ? RF(0.5) * dy[a] : r_fma(RF(0.5), dy[a], S0y[a]);
    }
    const real mqw = -qw;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        real acc = RF(0.0);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc = a ? r_fma(dx[a], sy[b], acc) : r_mul(dx[a], sy[b]);
            jput(col, a * 4 + b, r_mul(mqw, acc));
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const bool za = a == 0 || a == 3;
        real acc = RF(0.0);
        const real hdx = RF(0.5) * dx[a], hS0x = RF(0.5) * S0x[a];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            acc = b ? r_fma(dy[b], sx[a], acc) : r_mul(dy[b], sx[a]);
            jput(col, 12 + a * 3 + b, r_mul(mqw, acc));
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const bool zb = b == 0 || b == 3;
            // S0x S0y + dx/2 S0y + S0x/2 dy + dx dy / 3, without the terms that are zero
            const real dd3 = r_mul(dx[a], dy[b]);
            real w;
            if (za && zb) w = r_mul(dd3, RF(1.0) / RF(3.0));
            else if (za) w = r_fma(dd3, RF(1.0) / RF(3.0), r_mul(hdx, S0y[b]));
            else if (zb) w = r_fma(dd3, RF(1.0) / RF(3.0), r_mul(hS0x, dy[b]));
            else w = r_fma(dd3, RF(1.0) / RF(3.0), r_fma(hS0x, dy[b], r_fma(hdx, S0y[b], r_mul(S0x[a], S0y[b]))));
            jput(col, 24 + a * 4 + b, r_mul(qwbz, w));
        }
    }
}

// 1D: jx at 3 half nodes (0..2), jy (3..6), jz (7..10) at 4 nodes
__device__ __forceinline__ void esirkepov1_w(real x0, real x1, real qw, real qwby, real qwbz, real *col)
{
    real S0x[4], S1x[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) { S0x[a] = cic_w(x0, a - 1); S1x[a] = cic_w(x1, a - 1); }
    real acc_x = RF(0.0);
#pragma unroll
    for (int a = 0; a < 3; ++a) { acc_x += S1x[a] - S0x[a]; jput(col, a, -qw * acc_x); }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        real sv = RF(0.5) * (S0x[a] + S1x[a]);
        jput(col, 3 + a, qwby * sv);
        jput(col, 7 + a, qwbz * sv);
    }
}

__device__ __forceinline__ void jglobal(unsigned long long *J, real v)
{
    if (v != RF(0.0)) atomicAdd(J, (unsigned long long)fix40(v));
}

// The 3 x 3 grid points around cell (cx, cy) (columns cx-1..cx+1, rows
// cy-1..cy+1 wrapped in y; one row repeated in 1D) of the six field
// components, [component][row][column]: every CIC gather of a particle in
// the cell reads inside it.  Columns outside [0, nx] hold 0 (their weight is
// 0).  One warp fills it, 54 loads per cell instead of 24 per particle.
constexpr int TILE = 54;

template <int DIM, class Slab>
__device__ __forceinline__ void load_tile(real *tile, const Slab &S, const real *fe, const real *fb, int npts,
                                          int cx, int cy, int t0, int nt)
{
    const int W = S.nx + 1;
    for (int t = t0; t < TILE; t += nt) {
        const int comp = t / 9, r = (t % 9) / 3, l = t % 3;
        const int gx = cx - 1 + l;
        int gy = 0;
        if (DIM == 2) { gy = cy - 1 + r; gy = gy < 0 ? gy + S.ny : (gy >= S.ny ? gy - S.ny : gy); }
        const real *F = comp < 3 ? fe + (size_t)comp * npts : fb + (size_t)(comp - 3) * npts;
        tile[t] = (gx >= 0 && gx <= S.nx) ? __ldg(F + (size_t)gy * W + gx) : RF(0.0);
    }
}

// w0 (v0 f00 + v1 f10) + w1 (v0 f01 + v1 f11), its fused products written
// out (a particle's last bits must not depend on where it is inlined)
__device__ __forceinline__ real cic4(real w0, real w1, real v0, real v1, real f00, real f10, real f01, real f11)
{
    return r_fma(w0, r_fma(v0, f00, r_mul(v1, f10)), r_mul(w1, r_fma(v0, f01, r_mul(v1, f11))));
}

// the tile of a cell in shared memory
struct CellTile {
    const real *t;
    __device__ __forceinline__ real operator()(int comp, int r, int c) const { return t[comp * 9 + r * 3 + c]; }
};
// the same values read from the grid
struct GridTile {
    const real *fe, *fb;
    int npts, nx, ny, cx, cy;
    __device__ __forceinline__ real operator()(int comp, int r, int c) const
    {
        const int gx = cx - 1 + c;
        int gy = 0;
        if (ny > 1) { gy = cy - 1 + r; gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy); }
        const real *F = comp < 3 ? fe + (size_t)comp * npts : fb + (size_t)(comp - 3) * npts;
        return gx >= 0 && gx <= nx ? __ldg(F + (size_t)gy * (nx + 1) + gx) : RF(0.0);
    }
};

// component comp interpolated at tile columns x0, x0 + 1 and rows y0, y1
template <class Tile>
__device__ __forceinline__ real tinterp(const Tile &T, int comp, int x0, real w0, real w1, int y0, int y1, real v0,
                                        real v1)
{
    return cic4(w0, w1, v0, v1, T(comp, y0, x0), T(comp, y1, x0), T(comp, y0, x0 + 1), T(comp, y1, x0 + 1));
}

// One particle: gather from the tile of its cell, Boris, move; returns the
// next local cell, -1 when it left through an x boundary, -2 when its move
// is not finite.  ig: 1 / gamma after the push.
template <int DIM, class Slab, class Tile>
__device__ __forceinline__ int move_particle(const Slab &S, const Tile &tile, int cx, int cy, real xi, real eta,
                                             real &ux, real &uy, real &uz, real qm, real &xn, real &yn, real &ig)
{
    // node weights at columns cx, cx + 1; half nodes at cx - 1/2, cx + 1/2 or
    // cx + 1/2, cx + 3/2 (weight 0 beyond the slab); the same in y, periodic
    const bool hx = xi >= RF(0.5), hy = DIM == 2 && eta >= RF(0.5);
    const int hx0 = hx ? 1 : 0, hy0 = DIM == 2 ? (hy ? 1 : 0) : 1, hy1 = DIM == 2 ? hy0 + 1 : 1, ny1 = DIM == 2 ? 2 : 1;
    const real wn0 = RF(1.0) - xi, wn1 = xi;
    real wh1 = hx ? xi - RF(0.5) : xi + RF(0.5);
    real wh0 = RF(1.0) - wh1;
    if (!hx && cx == 0) wh0 = RF(0.0);
    if (hx && cx == S.nx - 1) wh1 = RF(0.0);
    real vn0 = RF(1.0), vn1 = RF(0.0), vh0 = RF(1.0), vh1 = RF(0.0);
    if (DIM == 2) {
        vn0 = RF(1.0) - eta; vn1 = eta;
        vh1 = hy ? eta - RF(0.5) : eta + RF(0.5);
        vh0 = RF(1.0) - vh1;
    }
    const real ex = tinterp(tile, 0, hx0, wh0, wh1, 1, ny1, vn0, vn1);
    const real ey = tinterp(tile, 1, 1, wn0, wn1, hy0, hy1, vh0, vh1);
    const real ez = tinterp(tile, 2, 1, wn0, wn1, 1, ny1, vn0, vn1);
    const real bx = tinterp(tile, 3, 1, wn0, wn1, hy0, hy1, vh0, vh1);
    const real by = tinterp(tile, 4, hx0, wh0, wh1, 1, ny1, vn0, vn1);
    const real bz = tinterp(tile, 5, hx0, wh0, wh1, hy0, hy1, vh0, vh1);
    boris(ux, uy, uz, ex, ey, ez, bx, by, bz, qm, S.dt);
    ig = r_rsqrt(r_fma(uz, uz, r_fma(uy, uy, r_fma(ux, ux, RF(1.0)))));
    const real c = (real)kCnmPerFs;
    xn = xi + r_mul(r_mul(r_mul(ux, ig), c), S.dt) / S.dx;
    yn = DIM == 2 ? eta + r_mul(r_mul(r_mul(uy, ig), c), S.dt) / S.dy : eta;
    if (!(r_fabs(xn - xi) < RF(64.0) && r_fabs(yn - eta) < RF(64.0))) return -2;
    real fx = r_floor(xn), fy = r_floor(yn);
    int ncx = cx + (int)fx;
    int ncy = DIM == 2 ? cy + (int)fy : 0;
    if (DIM == 2) { if (ncy < 0) ncy += S.ny; else if (ncy >= S.ny) ncy -= S.ny; }
    return (ncx < 0 || ncx >= S.nx) ? -1 : ncy * S.nx + ncx;
}

__device__ __forceinline__ void wrap_offsets(real xn, real yn, real &xi, real &eta)
{
    const real below1 = kBelow1;
    xi = xn - r_floor(xn);
    eta = yn - r_floor(yn);
    if (xi >= RF(1.0)) xi = below1;
    if (eta >= RF(1.0)) eta = below1;
}

// What the push needs of a slab's description, kept by each warp in shared
// memory: the stores of the particle loop make the compiler read it again
// for every batch, and registers are what limits the resident warps.
struct PushSlab {
    int nx, ny, cell0, fo, active;
    unsigned flags;
    real dt, dx, dy, w_ion, m_ion;
};

__device__ __forceinline__ PushSlab push_slab(const SlabDev &S)
{
    return PushSlab{S.nx, S.ny, S.cell0, S.fld_off, S.active, S.flags, S.dt, S.dx, S.dy, S.w_ion, S.m_ion};
}

// One batch: 32 particles of a species from position base of the cell.
// Every lane takes part (the row sums need all 32); t: the batch's current.
template <int DIM>
__device__ __forceinline__ void push_batch(const PushArgs &a, const PushSlab &S, int g, int cx, int cy, bool elec, int k0,
                                           int n, int base, int lane, real *sj, const real *tile, real (&t)[3])
{
    constexpr int NJ = DIM == 2 ? 40 : 11;
    const bool do_push = S.flags & 64u, do_dep = (S.flags & 128u) != 0;
    real4 *R0 = elec ? a.e0 : a.i0, *R1 = elec ? a.e1 : a.i1;
    const bool have = base + lane < n;
    const int k = k0 + base + lane;
    int nk = -1;
    real x0 = RF(0.5), y0 = RF(0.5), x1 = RF(0.5), y1 = RF(0.5), qw = RF(0.), qwby = RF(0.), qwbz = RF(0.);
    if (have) {
        const real4 P0 = R0[k], P1 = R1[k];
        if (elec ? P1.y <= RF(0.0) : (rec_ist(P1) & 0xff) == 0xff) {
            nk = -1;                                   // recombined away, or dropped
        } else if (!do_push) {
            nk = g;
        } else {
            const real q = elec ? -RF(1.0) : (real)(rec_ist(P1) & 0xff) + P1.y;
            const real m = elec ? RF(1.0) : S.m_ion, w = elec ? P1.y : S.w_ion;
            real xi = P0.x, eta = P0.y, ux = P0.z, uy = P0.w, uz = P1.x, xn, yn, ig;
            const int nc = move_particle<DIM>(S, CellTile{tile}, cx, cy, xi, eta, ux, uy, uz, q / m, xn, yn, ig);
            if (nc == -2) {
                nk = -1;
                atomicOr(a.err, ERR_NUMERIC);
            } else {
                if (do_dep) {
                    qw = q * w; qwby = qw * uy * ig; qwbz = qw * uz * ig;
                    if (r_fabs(xn - xi) < RF(1.0) && r_fabs(yn - eta) < RF(1.0)) {
                        x0 = xi; y0 = eta; x1 = xn; y1 = yn;
                    } else {
                        SlabGrid gr;
                        gr.nx = S.nx; gr.ny = S.ny; gr.W = S.nx + 1; gr.npts = a.npts; gr.fo = S.fo;
                        deposit_long(gr, a.J, a.npts, S.fo, cx, cy, xi, eta, xn, yn, qw, qwby, qwbz);
                        qw = qwby = qwbz = RF(0.0);
                    }
                }
                if (nc == -1) {                        // rare: tallied at once
                    const real4 Q0 = R0[k];
                    SlabTally *tl = a.tally + __ldg(a.cell_slab + g);
                    atomicAdd(&tl->esc, (double)(w * ((real)kMeC2 * m * gm1(Q0.z, Q0.w, R1[k].x))));
                    atomicAdd(tl->cnt + (elec ? C_ESC_E : C_ESC_I), 1ull);
                } else {
                    nk = S.cell0 + nc;
                }
                wrap_offsets(xn, yn, xi, eta);
                R0[k] = make_real4(xi, eta, ux, uy);
                reinterpret_cast<real *>(R1 + k)[0] = uz;
            }
        }
        (elec ? a.ekey : a.ikey)[k] = nk;
    }
    if (do_dep) {
        if constexpr (DIM == 2) esirkepov2_w(x0, y0, x1, y1, qw, qwbz, sj + lane);
        else esirkepov1_w(x0, x1, qw, qwby, qwbz, sj + lane);
        jrows<NJ>(sj, lane, t);
    }
    // aggregated count of the next cell
    unsigned peers = __match_any_sync(FULL, have ? nk : -2);
    if (have && nk >= 0 && lane == __ffs(peers) - 1) atomicAdd((elec ? a.cnt_e : a.cnt_i) + nk, __popc(peers));
}

// the total v of stencil row k of cell (cx, cy) to the global grid
template <int DIM>
__device__ __forceinline__ void deposit_row(const PushArgs &a, const PushSlab &S, int cx, int cy, int k, real v)
{
    int p, q = 0, comp;
    if (DIM == 2) {
        if (k < 12) { comp = 0; p = k / 4; q = k % 4; }
        else if (k < 24) { comp = 1; p = (k - 12) / 3; q = (k - 12) % 3; }
        else { comp = 2; p = (k - 24) / 4; q = (k - 24) % 4; }
    } else {
        if (k < 3) { comp = 0; p = k; } else if (k < 7) { comp = 1; p = k - 3; } else { comp = 2; p = k - 7; }
    }
    const int i = cx - 1 + p;
    int j = 0;
    if (DIM == 2) { j = cy - 1 + q; j = j < 0 ? j + S.ny : (j >= S.ny ? j - S.ny : j); }
    const bool ok = comp == 0 ? (i >= 0 && i < S.nx) : (i >= 0 && i <= S.nx);
    if (ok) jglobal(a.J + (size_t)comp * a.npts + S.fo + (size_t)j * (S.nx + 1) + i, v);
}

// The batches of a cell, electrons then ions, are numbered in a row; a
// team of TW warps takes TW of them a round, and their currents are added to
// the running totals in the order of their numbers.  tot: two rounds' batch
// currents of a team.
template <int DIM, int TW>
__device__ __forceinline__ void push_cell(const PushArgs &a, const PushSlab &S, int g, int warp, int lane, real *sj,
                                          real *tile, real *tot)
{
    constexpr int NJ = DIM == 2 ? 40 : 11, FULLROWS = NJ / 32 * 32;
    const int lc = g - S.cell0;
    const int cy = DIM == 2 ? lc / S.nx : 0, cx = lc - cy * S.nx;
    const bool do_dep = (S.flags & 128u) != 0;
    const int e0 = a.cs_e[g], ne = a.cs_e[g + 1] - e0, i0 = a.cs_i[g], ni = a.cs_i[g + 1] - i0;
    const int nbe = (ne + 31) >> 5, nb = nbe + ((ni + 31) >> 5);
    if (S.flags & 64u) {
        if (TW == 1) __syncwarp();
        load_tile<DIM>(tile, S, a.fldE + S.fo, a.fldB + S.fo, a.npts, cx, cy, warp * 32 + lane, 32 * TW);
        if (TW == 1) __syncwarp(); else __syncthreads();
    }
    real acc[3] = {RF(0.0), RF(0.0), RF(0.0)};
    for (int b0 = 0, par = 0; b0 < nb; b0 += TW, par ^= 1) {
        const int b = b0 + warp;
        real t[3] = {RF(0.0), RF(0.0), RF(0.0)};
        if (TW == 1 || b < nb) {
            const bool elec = b < nbe;
            push_batch<DIM>(a, S, g, cx, cy, elec, elec ? e0 : i0, elec ? ne : ni, 32 * (elec ? b : b - nbe), lane, sj,
                            tile, t);
        }
        if (!do_dep) continue;
        if constexpr (TW == 1) {
#pragma unroll
            for (int h = 0; h < 3; ++h) acc[h] += t[h];
        } else {
            real *row = tot + (par * TW + warp) * NJ;
            if (FULLROWS > 0) row[lane] = t[0];
#pragma unroll
            for (int h = 0; FULLROWS + 8 * h < NJ; ++h) {
                const int k = FULLROWS + 8 * h + (lane >> 2);
                if (k < NJ && (lane & 3) == 0) row[k] = t[1 + h];
            }
            __syncthreads();
            const int k = warp * 32 + lane;
            if (k < NJ)
                for (int w = 0; w < TW; ++w) acc[0] += tot[(par * TW + w) * NJ + k];
        }
    }
    if (!do_dep) return;
    if constexpr (TW == 1) {
        if (FULLROWS > 0) deposit_row<DIM>(a, S, cx, cy, lane, acc[0]);
#pragma unroll
        for (int h = 0; FULLROWS + 8 * h < NJ; ++h) {
            const int k = FULLROWS + 8 * h + (lane >> 2);
            if (k < NJ && (lane & 3) == 0) deposit_row<DIM>(a, S, cx, cy, k, acc[1 + h]);
        }
    } else {
        const int k = warp * 32 + lane;
        if (k < NJ) deposit_row<DIM>(a, S, cx, cy, k, acc[0]);
    }
}

// The first records of a cell (96 electrons, 32 ions, a line a lane) into
// L2, for the warp that will take it about one cell's time from now: the
// cells are handed out in order, so that is a grid's worth of warps ahead.
__device__ __forceinline__ void prefetch_cell(const PushArgs &a, int g, int lane)
{
    constexpr int PER = 128 / sizeof(real4);
    if (g >= a.ncell) return;
    const bool elec = lane < 24;
    const int *cs = elec ? a.cs_e : a.cs_i;
    const int q = elec ? lane % 12 : lane % 4, k = cs[g] + PER * q;
    if (k >= cs[g + 1]) return;
    const bool first = elec ? lane < 12 : lane < 28;
    prefetch_l2((elec ? (first ? a.e0 : a.e1) : (first ? a.i0 : a.i1)) + k);
}

// An electron created this step: they sit after the sorted range with their
// cell in the key; each is pushed by one thread and deposits straight to the
// global grid (integer atomics, so the order does not matter).
__device__ __noinline__ void push_new(const PushArgs &a, int k)
{
    const int g = a.ekey[k];
    if (g < 0) return;
    const int s = __ldg(a.cell_slab + g);
    const PushSlab S = push_slab(a.slabs[s]);
    const int lc = g - S.cell0, cx = lc % S.nx, cy = lc / S.nx;
    const real4 P0 = a.e0[k], P1 = a.e1[k];
    int nk = g;
    if (S.flags & 64u) {
        const GridTile T{a.fldE + S.fo, a.fldB + S.fo, a.npts, S.nx, S.ny, cx, cy};
        real xi = P0.x, eta = P0.y, ux = P0.z, uy = P0.w, uz = P1.x, xn, yn, ig;
        const real ke = (real)kMeC2 * gm1(ux, uy, uz);
        const int nc = S.ny > 1 ? move_particle<2>(S, T, cx, cy, xi, eta, ux, uy, uz, -RF(1.0), xn, yn, ig)
                                : move_particle<1>(S, T, cx, cy, xi, eta, ux, uy, uz, -RF(1.0), xn, yn, ig);
        if (nc == -2) {
            nk = -1;
            atomicOr(a.err, ERR_NUMERIC);
        } else {
            if (S.flags & 128u) {
                const real qw = -P1.y;
                SlabGrid gr;
                gr.nx = S.nx; gr.ny = S.ny; gr.W = S.nx + 1; gr.npts = a.npts; gr.fo = S.fo;
                deposit_long(gr, a.J, a.npts, S.fo, cx, cy, xi, eta, xn, yn, qw, qw * uy * ig, qw * uz * ig);
            }
            if (nc == -1) {
                nk = -1;
                atomicAdd(&a.tally[s].esc, (double)(P1.y * ke));
                atomicAdd(a.tally[s].cnt + C_ESC_E, 1ull);
            } else {
                nk = S.cell0 + nc;
            }
            wrap_offsets(xn, yn, xi, eta);
            a.e0[k] = make_real4(xi, eta, ux, uy);
            reinterpret_cast<real *>(a.e1 + k)[0] = uz;
        }
    }
    a.ekey[k] = nk;
    if (nk >= 0) atomicAdd(a.cnt_e + nk, 1);
}

__device__ __forceinline__ void push_created(const PushArgs &a, int t0, int nt)
{
    const int sorted = a.cs_e[a.ncell], n = min(*a.append, a.cap_e - sorted);
    for (int t = t0; t < n; t += nt) push_new(a, sorted + t);
}

// One warp per cell, cells handed out from a counter.  Bound by the latency
// of dependent loads and arithmetic (14 % of DRAM throughput at 16 warps an
// SM).  The stencil rows are 48 KB a CTA, so four are resident, 32 warps an SM:
// the bound of five in 2D is there for its register cap (48).  2048 x 256
// cells, 42 M particles, a step: 2.90 ms with scalar reads of the stencil
// rows, all 40 weights formed from four-node shapes and 16 warps an SM; 1.82
// ms with 16-byte row reads, the weights that are zero left out, the next
// cell's records prefetched and four CTAs an SM at 48 registers, spills included
// (64 registers, the bound of four: 2.00 ms; 40, the bound of six: 1.86).
// In 1D, with a quarter of the stencil's arithmetic, two CTAs without spills
// are faster.
template <int DIM>
__global__ void __launch_bounds__(32 * PUSH_WARPS, DIM == 2 ? 5 : 2) k_push(PushArgs a)
{
    __shared__ JStage s_j[PUSH_WARPS];
    __shared__ real s_t[PUSH_WARPS][TILE];
    __shared__ PushSlab s_slab[PUSH_WARPS];
    const int lane = threadIdx.x & 31;
    real *sj = s_j[threadIdx.x >> 5].v;
    real *tile = s_t[threadIdx.x >> 5];
    PushSlab &S = s_slab[threadIdx.x >> 5];
    push_created(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
    int cur = -1;
    for (;;) {
        int g = 0;
        if (lane == 0) g = atomicAdd(a.work, 1);
        g = __shfl_sync(FULL, g, 0);
        if (g >= a.ncell) break;
        prefetch_cell(a, g + (int)(gridDim.x * PUSH_WARPS), lane);
        if (a.cs_e[g + 1] == a.cs_e[g] && a.cs_i[g + 1] == a.cs_i[g]) continue;
        const int s = __ldg(a.cell_slab + g);
        if (s != cur) {
            cur = s;
            __syncwarp();
            if (lane == 0) S = push_slab(a.slabs[s]);
            __syncwarp();
        }
        if (!S.active) {              // retired slab: its particles leave
            for (int k = a.cs_e[g] + lane; k < a.cs_e[g + 1]; k += 32) a.ekey[k] = -1;
            for (int k = a.cs_i[g] + lane; k < a.cs_i[g + 1]; k += 32) a.ikey[k] = -1;
            continue;
        }
        push_cell<DIM, 1>(a, S, g, 0, lane, sj, tile, nullptr);
    }
}

// One cell per block of TW warps: for contexts with few cells, whose batches
// one warp would take one after another (128 cells of 320 particles: 36 ->
// 15 us a step with the created electrons, which had a launch of their own;
// 700 of 920: 65 -> 33 us).  The first PUSH_NEW_CTAS blocks take the created
// electrons.
template <int DIM, int TW>
__global__ void __launch_bounds__(32 * TW, 4) k_push_team(PushArgs a)
{
    __shared__ JStage s_j[TW];
    __shared__ real s_t[TILE], s_tot[2 * TW * JROWS];
    __shared__ PushSlab S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = (int)blockIdx.x - PUSH_NEW_CTAS;
    if (g < 0) {
        push_created(a, blockIdx.x * blockDim.x + threadIdx.x, PUSH_NEW_CTAS * blockDim.x);
        return;
    }
    const int e0 = a.cs_e[g], e1 = a.cs_e[g + 1], i0 = a.cs_i[g], i1 = a.cs_i[g + 1];
    if (e0 == e1 && i0 == i1) return;
    if (threadIdx.x == 0) S = push_slab(a.slabs[__ldg(a.cell_slab + g)]);
    __syncthreads();
    if (!S.active) {              // retired slab: its particles leave
        for (int k = e0 + threadIdx.x; k < e1; k += 32 * TW) a.ekey[k] = -1;
        for (int k = i0 + threadIdx.x; k < i1; k += 32 * TW) a.ikey[k] = -1;
        return;
    }
    push_cell<DIM, TW>(a, S, g, warp, lane, s_j[warp].v, s_t, s_tot);
}

}  // namespace pic
