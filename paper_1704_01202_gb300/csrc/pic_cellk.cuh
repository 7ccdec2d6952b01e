// The per-cell collision and atomic-process kernel k_cell: one warp, or a
// block of four, per cell (see pic_cell.cuh for the building blocks; the
// push and deposit follow in pic_push.cuh).
#pragma once
#include <type_traits>
#include "pic_cell.cuh"

namespace pic {

// event counts and energy tallies of one warp, lane-uniform, flushed to the
// slab's tally when the warp moves to another slab and at the end
struct WarpTally {
    int slab;
    dd ion, ka, esc;
    dd rt;          // energy the electrons took from the radiation field (transport mode)
    int cnt[NCOUNT];
};

// the counts every cell adds to, kept per lane and summed at the flush
struct LaneTally { int ee, ei, ion, rej; };

__device__ __forceinline__ void tally_flush(const CellArgs &a, WarpTally &w, LaneTally &l, int lane)
{
    w.cnt[C_EE] += wsum_i(l.ee);
    w.cnt[C_EI] += wsum_i(l.ei);
    w.cnt[C_ION] += wsum_i(l.ion);
    w.cnt[C_ION_REJ] += wsum_i(l.rej);
    l = LaneTally{0, 0, 0, 0};
    if (w.slab >= 0 && lane == 0) {
        SlabTally *tl = a.tally + w.slab;
        if (dd_f(w.ion) != RF(0.0)) atomicAdd(&tl->ion, (double)w.ion.hi + (double)w.ion.lo);
        if (dd_f(w.ka) != RF(0.0)) atomicAdd(&tl->ka_esc, (double)w.ka.hi + (double)w.ka.lo);
        if (dd_f(w.esc) != RF(0.0)) atomicAdd(&tl->esc, (double)w.esc.hi + (double)w.esc.lo);
        if (dd_f(w.rt) != RF(0.0)) atomicAdd(&tl->rt_pend, -((double)w.rt.hi + (double)w.rt.lo));
        for (int q = 0; q < NCOUNT; ++q)
            if (w.cnt[q]) atomicAdd(tl->cnt + q, (unsigned long long)w.cnt[q]);
    }
    w.ion = w.ka = w.esc = w.rt = dd_zero();
    for (int q = 0; q < NCOUNT; ++q) w.cnt[q] = 0;
}

// per-cell scalars of the out-of-line stages
struct CellCtx {
    int lc, ne, ni;
    unsigned step;
    unsigned long long seed;
    real wi, n_i, nref;
    // sums the recombination stage needs, when the earlier stages already
    // hold them (every electron bulk, impact ionization run): kinetic
    // energy of the electrons after the ionization payment, their weight,
    // and the ion charge after ionization
    bool have_sums;
    dd K_after;
    real W_e, Q_after;
};

// ---- forced-thermalization variant (Sec. VI C), rad steps ----
// The cell's free electrons, those created in this step included, are
// redrawn from a Maxwellian at kT = (2/3) E_ave (components normal with
// standard deviation sqrt(kT / m c^2), Box-Muller on the electron's Philox
// draw); the mean momentum is shifted back to the cell's and the momenta
// about it scaled by one factor (Newton) so that the cell's kinetic energy
// is kept.  Sums are double-float (double-double in the FP64 build).
__device__ __forceinline__ real gm1_free(real ux, real uy, real uz)
{
    return gm1_of(ux * ux + uy * uy + uz * uz);
}

struct ThermSums { dd W, K, Px, Py, Pz; int n; };

__device__ __forceinline__ void therm_add(ThermSums &t, real4 u)
{
    t.W = dd_addf(t.W, u.w);
    t.K = dd_addf(t.K, u.w * (real)kMeC2 * gm1_free(u.x, u.y, u.z));
    t.Px = dd_addf(t.Px, u.w * u.x); t.Py = dd_addf(t.Py, u.w * u.y); t.Pz = dd_addf(t.Pz, u.w * u.z);
    t.n += 1;
}

__device__ __noinline__ void stage_therm(const CellMem &m, const CellCtx &c, int lane, int nnew)
{
    const int ne = c.ne;
    const real MC2 = (real)kMeC2;
    ThermSums t0{dd_zero(), dd_zero(), dd_zero(), dd_zero(), dd_zero(), 0};
    for (int k = lane; k < ne; k += 32) { real4 u = m.eu[k]; if (u.w > RF(0.0)) therm_add(t0, u); }
    for (int k = lane; k < nnew; k += 32) {
        NewE q = m.nw[k];
        if (q.w > RF(0.0)) therm_add(t0, make_real4(q.ux, q.uy, q.uz, q.w));
    }
    const dd W = wsum_dd(t0.W), K = wsum_dd(t0.K);
    const real P[3] = {dd_f(wsum_dd(t0.Px)), dd_f(wsum_dd(t0.Py)), dd_f(wsum_dd(t0.Pz))};
    const int n = wsum_i(t0.n);
    const real Wf = dd_f(W), Kf = dd_f(K);
    if (n < 2 || !(Wf > RF(0.0)) || !(Kf > RF(0.0))) return;
    const real sig = r_sqrt((RF(2.0) / RF(3.0)) * Kf / Wf / MC2);
    // redraw; the new momenta replace the old ones in shared memory
    auto redraw = [&](unsigned long long id) {
        U4 r = draw(c.seed, id, c.step, PU_THERM);
        const real a0 = r_sqrt(-RF(2.0) * r_log(u01(r.x))), a1 = r_sqrt(-RF(2.0) * r_log(u01(r.z)));
        real sn, cs;
        r_sincos(RF(2.0) * kPiR * u01(r.y), &sn, &cs);
        return make_real3(sig * a0 * cs, sig * a0 * sn, sig * a1 * r_cos(RF(2.0) * kPiR * u01(r.w)));
    };
    dd Qx = dd_zero(), Qy = dd_zero(), Qz = dd_zero();
    for (int k = lane; k < ne; k += 32) {
        real4 u = m.eu[k];
        if (!(u.w > RF(0.0))) continue;
        real3 v = redraw(m.eid[k]);
        m.eu[k] = make_real4(v.x, v.y, v.z, u.w);
        Qx = dd_addf(Qx, u.w * v.x); Qy = dd_addf(Qy, u.w * v.y); Qz = dd_addf(Qz, u.w * v.z);
    }
    for (int k = lane; k < nnew; k += 32) {
        NewE q = m.nw[k];
        if (!(q.w > RF(0.0))) continue;
        const int islot = q.meta & 0xffff, kind = q.meta >> 16;
        const unsigned ion_id = m.iid[islot];
        const unsigned long long id = ((unsigned long long)(((c.step + 1u) << 2) | (unsigned)kind) << 32) | ion_id;
        real3 v = redraw(id);
        q.ux = v.x; q.uy = v.y; q.uz = v.z;
        m.nw[k] = q;
        Qx = dd_addf(Qx, q.w * v.x); Qy = dd_addf(Qy, q.w * v.y); Qz = dd_addf(Qz, q.w * v.z);
    }
    __syncwarp();
    const real iW = RF(1.0) / Wf;
    const real V[3] = {P[0] * iW, P[1] * iW, P[2] * iW};
    const real M[3] = {dd_f(wsum_dd(Qx)) * iW, dd_f(wsum_dd(Qy)) * iW, dd_f(wsum_dd(Qz)) * iW};
    // kinetic energy of the cell with the peculiar momenta d = u - M scaled by s
    auto energy = [&](real s, real &slope) {
        dd e = dd_zero(), de = dd_zero();
        auto one = [&](real4 u) {
            real dx = u.x - M[0], dy = u.y - M[1], dz = u.z - M[2];
            real ux = V[0] + s * dx, uy = V[1] + s * dy, uz = V[2] + s * dz;
            e = dd_addf(e, u.w * MC2 * gm1_free(ux, uy, uz));
            de = dd_addf(de, u.w * MC2 * (ux * dx + uy * dy + uz * dz) * r_rsqrt(RF(1.0) + ux * ux + uy * uy + uz * uz));
        };
        for (int k = lane; k < ne; k += 32) { real4 u = m.eu[k]; if (u.w > RF(0.0)) one(u); }
        for (int k = lane; k < nnew; k += 32) {
            NewE q = m.nw[k];
            if (q.w > RF(0.0)) one(make_real4(q.ux, q.uy, q.uz, q.w));
        }
        slope = dd_f(wsum_dd(de));
        return wsum_dd(e);
    };
    real s = RF(1.0);
    for (int it = 0; it < 8; ++it) {
        real slope;
        const dd e = energy(s, slope);
        if (!(slope > RF(0.0))) break;
        const real ds = dd_f(dd_sub(e, K)) / slope;
        s = r_fmax(s - ds, RF(0.0));
        if (r_fabs(ds) <= RF(1e-7) * s) break;
    }
    for (int k = lane; k < ne; k += 32) {
        real4 u = m.eu[k];
        if (!(u.w > RF(0.0))) continue;
        m.eu[k] = make_real4(V[0] + s * (u.x - M[0]), V[1] + s * (u.y - M[1]), V[2] + s * (u.z - M[2]), u.w);
    }
    for (int k = lane; k < nnew; k += 32) {
        NewE q = m.nw[k];
        if (!(q.w > RF(0.0))) continue;
        q.ux = V[0] + s * (q.ux - M[0]); q.uy = V[1] + s * (q.uy - M[1]); q.uz = V[2] + s * (q.uz - M[2]);
        m.nw[k] = q;
    }
    __syncwarp();
}

// ---- EOS-clamped three-body recombination (Sec. IV) ----
// How many events the clamp asks for, before what the cell can give; Wex:
// the electrons' weight.  By one warp.
__device__ __forceinline__ int recombine_wanted(const CellArgs &a, const CellMem &m, real E_bulk, const CellCtx &c, int lane,
                                                real Wnew_imp, real &Wex)
{
    const int ne = c.ne, ni = c.ni;
    const real MC2 = (real)kMeC2;
    real zb, Wb2, Kb2;
    if (c.have_sums) {
        // every electron is bulk: the sums of the moments and ionization
        // stages, which the ionization payment changed by a known amount
        zb = c.Q_after / ni;
        Wb2 = c.W_e + Wnew_imp;
        Kb2 = dd_f(c.K_after);
        Wex = c.W_e;
    } else {
        real pq = RF(0.0);
        for (int k = lane; k < ni; k += 32) pq += (real)(m.ist[k] & 0xff) + m.iu[k].w;
        zb = wsum_f(pq) / ni;
        dd pkb = dd_zero();
        real pwb = RF(0.0), pwx = RF(0.0);
        for (int k = lane; k < ne; k += 32) {
            real4 u = m.eu[k];
            real ke = MC2 * gm1(u.x, u.y, u.z);
            pwx += u.w;
            if (E_bulk <= RF(0.0) || ke < E_bulk) { pwb += u.w; pkb = dd_addf(pkb, u.w * ke); }
        }
        Wb2 = wsum_f(pwb) + Wnew_imp;
        Kb2 = dd_f(wsum_dd(pkb));
        Wex = wsum_f(pwx);
    }
    const real Te2 = Wb2 > RF(0.0) ? (RF(2.0) / RF(3.0)) * Kb2 / Wb2 : RF(0.0);
    const real zeos = eos_lookup(*a.eos, c.n_i, Te2, lane);
    return zb > zeos ? (int)r_floor((zb - zeos) * ni + RF(0.5)) : 0;
}

// The events themselves (in a fifth of the cells of a solid-density plasma,
// so out of line), by one warp; a team's other warps join for the last pass,
// the correction of every electron's energy (recombine_apply).  Returns
// whether events happened, with that pass's factor in delta.
__device__ __noinline__ bool stage_recombine(const CellArgs &a, const CellMem &m, const Tables &T, real E_bulk, real wi,
                                             int ne, int ni, int lane, int Kev, real Wex, WarpTally &wt, real &delta)
{
    const real MC2 = (real)kMeC2;
    int pel = 0;
    for (int k = lane; k < ni; k += 32) pel += m.ist[k] & 0xff;
    const int elig = wsum_i(pel);
    Kev = min(Kev, elig);
    Kev = min(Kev, (int)r_floor(Wex / wi * (RF(1.0) + RF(1e-6))));
    if (Kev <= 0) return false;
    int *nrec = m.nrec;
    real *take = (real *)m.ew;
    for (int k = lane; k < ni; k += 32) nrec[k] = 0;
    __syncwarp();
    int left = Kev;
    for (int round = 0; left > 0; ++round) {
        if (round > ZNUC * 2) {          // cannot happen when Kev <= sum Z
            if (lane == 0) atomicOr(a.err, ERR_NUMERIC);
            break;
        }
        for (int b0 = 0; b0 < ni && left > 0; b0 += 32) {
            int t = b0 + lane;
            bool e = false;
            if (t < ni) e = (m.ist[t] & 0xff) - nrec[t] >= 1;
            unsigned bal = __ballot_sync(FULL, e);
            int rank = __popc(bal & ((1u << lane) - 1u));
            if (e && rank < left) nrec[t] += 1;
            left -= min(left, __popc(bal));
            __syncwarp();
        }
    }
    // the electron weight removed, in canonical order: once the weight
    // passed is beyond it by more than rounding, the rest give nothing
    // (weights are not negative)
    const dd Wrem = dd{(real)Kev * wi, RF(0.0)};
    dd carry = dd_zero(), remKE = dd_zero();
    bool more = true;
    for (int b0 = 0; b0 < ne; b0 += 32) {
        int t = b0 + lane;
        if (!more) {
            if (t < ne) take[t] = RF(0.0);
            continue;
        }
        real w = RF(0.0), ke = RF(0.0);
        if (t < ne) { real4 u = m.eu[t]; w = u.w; ke = MC2 * gm1(u.x, u.y, u.z); }
        dd incl = dd_add(carry, wscan_dd(dd{w, RF(0.0)}, lane));
        dd before = dd_sub(incl, dd{w, RF(0.0)});
        real tk = r_fmin(r_fmax(dd_f(dd_sub(Wrem, before)), RF(0.0)), w);
        if (t < ne) take[t] = tk;
        remKE = dd_addf(remKE, tk * ke);
        carry = wlane_dd(incl, 31);
        more = !(dd_f(dd_sub(Wrem, carry)) < -RF(1e-6) * Wrem.hi);
    }
    __syncwarp();
    remKE = wsum_dd(remKE);
    dd pb = dd_zero();
    for (int k = lane; k < ni; k += 32) {
        int st = m.ist[k];
        int Z = st & 0xff, nK = (st >> 8) & 0xff;
        for (int r = 1; r <= nrec[k]; ++r) pb = dd_addf(pb, wi * removal_energy(T, Z - r, nK, m.dE[Z - r]));
    }
    const dd bind = wsum_dd(pb);
    dd pkr = dd_zero();
    for (int k = lane; k < ne; k += 32) {
        real4 u = m.eu[k];
        real ke = MC2 * gm1(u.x, u.y, u.z);
        if (E_bulk <= RF(0.0) || ke < E_bulk) pkr = dd_addf(pkr, (u.w - take[k]) * ke);
    }
    const real Krem = dd_f(wsum_dd(pkr));
    if (!(Krem > RF(0.0))) return false;
    delta = -dd_f(dd_add(remKE, bind)) / Krem;
    for (int k = lane; k < ni; k += 32) m.ist[k] = m.ist[k] - nrec[k];
    wt.ion = dd_sub(wt.ion, bind);
    wt.cnt[C_REC] += Kev;
    __syncwarp();
    return true;
}

__device__ __forceinline__ void recombine_apply(const CellMem &m, const SlabDev &S, int ne, real delta, int t, int nt)
{
    const real *take = (const real *)m.ew;
    const real E_bulk = S.E_bulk;
    for (int k = t; k < ne; k += nt) {
        real4 u = m.eu[k];
        real ke = (real)kMeC2 * gm1(u.x, u.y, u.z);
        bool bulk = E_bulk <= RF(0.0) || ke < E_bulk;
        real tk = take[k];
        real wn = u.w - tk;
        bool dead = tk > RF(0.0) && wn <= RF(0.0);
        u.w = dead ? RF(0.0) : wn;
        if (bulk && !dead) scale_kinetic(u.x, u.y, u.z, delta);
        m.eu[k] = u;
    }
}

// ---- rad step: subshell photoionization (Eq. 2) ----
__device__ __noinline__ void stage_photo(const CellArgs &a, const CellMem &m, const Tables &T, const SlabDev &S,
                                         const CellCtx &c, int lane, int &nnew, WarpTally &wt)
{
    const int ni = c.ni, nb = S.nb;
    const real wi = c.wi;
    const real dtr = S.rad_every * S.dt;
    ph2 *ph = a.photons + S.ph_off + (size_t)c.lc * nb;
    dd *n0 = m.ph, *used = m.ph + MAXB;
    int *carry = m.phc;
    if (lane < nb) { ph2 v = ph[lane]; n0[lane] = dd{v.hi, v.lo}; used[lane] = dd_zero(); carry[lane] = 0; }
    __syncwarp();
    const real cph = (real)kCcmPerFs * dtr * c.nref;
    int c_part = 0, c_ph[NS] = {0, 0, 0, 0, 0};
    // transport mode: the ions' opacity per bin (sum over occupied subshells
    // of N_s sigma_s above the lowered edge) and the photon energy the
    // events take; the field is not depleted here (its opacity does that)
    const bool rtm = S.rt != 0;
    real chi_l[MAXB];
    for (int b = 0; b < MAXB; ++b) chi_l[b] = RF(0.0);
    dd emc = dd_zero();
    for (int b0 = 0; b0 < ni; b0 += 32) {
        int t = b0 + lane;
        int sub = -1, bin = -1, sl = 0, Z = 0, nK = 0;
        real edge = RF(0.), rc = RF(0.), rp = RF(0.);
        if (t < ni) {
            sl = t;
            int st = m.ist[sl];
            Z = st & 0xff; nK = (st >> 8) & 0xff;
            int occ[NS];
            if (Z < ZNUC && occupancy(ZNUC - Z, nK, occ)) {
                if (rtm)
                    for (int q = 0; q < NS; ++q) {
                        if (!occ[q]) continue;
                        const real ed = lowered_binding(T, Z, q, m.dE[Z]);
                        for (int b = 0; b < nb; ++b)
                            if (S.hv_b[b] > ed) chi_l[b] += (real)occ[q] * S.sig_b[q][b];
                    }
                U4 ra = draw(c.seed, (unsigned long long)m.iid[t], c.step, PU_PHOTO_A);
                U4 rb = draw(c.seed, (unsigned long long)m.iid[t], c.step, PU_PHOTO_B);
                real rs[NS] = {u01(ra.x), u01(ra.y), u01(ra.z), u01(ra.w), u01(rb.x)};
                real Ps = RF(0.);
                for (int q = 0; q < NS; ++q) {
                    if (!occ[q]) continue;
                    real ed = lowered_binding(T, Z, q, m.dE[Z]);
                    real acc = RF(0.);
                    for (int b = 0; b < nb; ++b)
                        if (S.hv_b[b] > ed) acc += dd_f(n0[b]) * S.sig_b[q][b];
                    real P = cph * occ[q] * acc;
                    if (rs[q] < P) { sub = q; Ps = P; edge = ed; break; }
                }
                if (sub >= 0) {
                    real target = u01(rb.y) * Ps, cum = RF(0.);
                    int lastpos = -1;
                    for (int b = 0; b < nb; ++b) {
                        real cb = S.hv_b[b] > edge ? cph * occ[sub] * dd_f(n0[b]) * S.sig_b[sub][b] : RF(0.);
                        if (cb > RF(0.)) lastpos = b;
                        cum += cb;
                        if (cum > target) { bin = b; break; }
                    }
                    if (bin < 0) bin = lastpos;
                    rc = u01(rb.z); rp = u01(rb.w);
                }
            }
        }
        // the k-th event of a bin gets min(w, max(0, n_bin - k w)) photons
        real g = RF(0.0);
        bool full = false;
        for (int b = 0; b < nb; ++b) {
            bool eb = bin == b && sub >= 0;
            unsigned bal = __ballot_sync(FULL, eb);
            if (eb) {
                int rank = carry[b] + __popc(bal & ((1u << lane) - 1u));
                dd rest = dd_addf(n0[b], -(real)rank * wi);
                if (dd_le(dd{wi, RF(0.0)}, rest)) { g = wi; full = true; }
                else g = r_fmax(dd_f(rest), RF(0.0));
            }
            __syncwarp();
            if (lane == 0) carry[b] += __popc(bal);
            __syncwarp();
        }
        bool ev = sub >= 0 && bin >= 0 && g > RF(0.0);
        if (ev) {
            if (full) {
                lose_electron(Z, nK, sub);
            } else {
                real zf = m.iu[sl].w + g / wi;
                if (zf >= RF(1.0)) {
                    zf -= RF(1.0);
                    int so = outer_shell(ZNUC - Z, nK);
                    if (so >= 0) lose_electron(Z, nK, so);
                }
                m.iu[sl].w = zf;
                c_part++;
            }
            m.ist[sl] = Z | (nK << 8);
            c_ph[sub]++;
        }
        for (int b = 0; b < nb; ++b) {
            dd ub = wsum_dd(dd{ev && bin == b ? g : RF(0.0), RF(0.0)});
            if (lane == 0) used[b] = dd_add(used[b], ub);
        }
        wt.ion = dd_add(wt.ion, wsum_dd(dd{ev ? g * edge : RF(0.0), RF(0.0)}));
        if (rtm) emc = dd_add(emc, wsum_dd(dd{ev ? g * S.hv_b[bin] : RF(0.0), RF(0.0)}));
        unsigned bal = __ballot_sync(FULL, ev);
        if (ev) {
            int pos = nnew + __popc(bal & ((1u << lane) - 1u));
            if (pos < a.cap_new) {
                real3 u = iso_momentum(S.hv_b[bin] - edge, rc, rp);
                NewE q; q.ux = u.x; q.uy = u.y; q.uz = u.z; q.w = g;
                q.meta = sl | (KIND_PHOTO << 16);
                m.nw[pos] = q;
            } else {
                atomicOr(a.err, ERR_NEW_OVERFLOW);
            }
        }
        nnew = min(nnew + __popc(bal), a.cap_new);
        __syncwarp();
    }
    if (rtm) {
        // opacity (cm^-1) and the events' photon energy, owed to the field
        // until its opacity takes it at the next transport step
        for (int b = 0; b < nb; ++b) {
            const real v = wsum_f(chi_l[b]);
            if (lane == 0) S.rt_chi[(size_t)c.lc * nb + b] = (float)(v * c.nref * c.wi);
        }
        if (lane == 0) S.rt_emc[c.lc] = (double)emc.hi + (double)emc.lo;
        wt.rt = dd_add(wt.rt, emc);
    } else if (lane < nb) {
        dd r = dd_sub(n0[lane], used[lane]);
        ph[lane] = ph2{r.hi, r.lo};
    }
    wt.cnt[C_PART] += wsum_i(c_part);
    for (int q = 0; q < NS; ++q) wt.cnt[C_PH0 + q] += wsum_i(c_ph[q]);
    __syncwarp();
}

// ---- rad step: K-vacancy decay with KLL Auger / K-alpha branching ----
__device__ __noinline__ void stage_decay(const CellArgs &a, const CellMem &m, const Tables &T, const SlabDev &S,
                                         const CellCtx &c, int lane, int &nnew, WarpTally &wt)
{
    const int ni = c.ni, nb = S.nb;
    const real wi = c.wi;
    const real dtr = S.rad_every * S.dt;
    dd *addph = m.ph;
    if (lane < MAXB) addph[lane] = dd_zero();
    __syncwarp();
    int c_aug = 0, c_ka = 0;
    for (int b0 = 0; b0 < ni; b0 += 32) {
        int t = b0 + lane;
        int kind = 0, sl = 0, Z = 0;
        real EA = RF(0.), rc = RF(0.), rp = RF(0.), Eka = RF(0.);
        if (t < ni) {
            sl = t;
            int st = m.ist[sl];
            Z = st & 0xff;
            int nK = (st >> 8) & 0xff;
            int nbd = ZNUC - Z, occ[NS];
            if (nK > 0 && occupancy(nbd, nK, occ)) {
                real tau = T.tauK[nbd][nK - 1];
                if (tau > RF(0.)) {
                    U4 r = draw(c.seed, (unsigned long long)m.iid[t], c.step, PU_DECAY);
                    if (u01(r.x) < dtr / tau) {
                        real om = T.omegaK[nbd][nK - 1];
                        int nl = occ[1] + occ[2];
                        if (u01(r.y) < RF(1.0) - om) {
                            if (nl >= 2) {
                                real e2s = lowered_binding(T, Z, 1, m.dE[Z]);
                                real e2p = lowered_binding(T, Z, 2, m.dE[Z]);
                                EA = r_fmax(T.E_Ka[Z] - (occ[1] * e2s + occ[2] * e2p) / nl, RF(0.0));
                                int kocc = occ[0] + 1, nb2 = nbd - 1;
                                int Zn = Z + 1, nKn = (nb2 < 2 ? nb2 : 2) - kocc;
                                m.ist[sl] = Zn | (nKn << 8);
                                kind = 1;
                                rc = u01(r.z); rp = u01(r.w);
                            }
                        } else if (occ[2] >= 1) {
                            Eka = T.E_Ka[Z];
                            m.ist[sl] = Z | ((nK - 1) << 8);
                            kind = 2;
                        }
                    }
                }
            }
        }
        unsigned bal = __ballot_sync(FULL, kind == 1);
        if (kind == 1) {
            int pos = nnew + __popc(bal & ((1u << lane) - 1u));
            if (pos < a.cap_new) {
                real3 u = iso_momentum(EA, rc, rp);
                NewE q; q.ux = u.x; q.uy = u.y; q.uz = u.z; q.w = wi; q.meta = sl | (KIND_AUGER << 16);
                m.nw[pos] = q;
            } else {
                atomicOr(a.err, ERR_NEW_OVERFLOW);
            }
            c_aug++;
        }
        nnew = min(nnew + __popc(bal), a.cap_new);
        int hit = -1;
        if (kind == 2) {
            c_ka++;
            for (int b = 0; b < nb; ++b)
                if (Eka >= S.hv_b[b] - S.bin_hw && Eka < S.hv_b[b] + S.bin_hw) { hit = b; break; }
        }
        for (int b = 0; b < nb; ++b) {
            dd v = wsum_dd(dd{hit == b ? wi * Eka / S.hv_b[b] : RF(0.0), RF(0.0)});
            if (lane == 0) addph[b] = dd_add(addph[b], v);
        }
        wt.ka = dd_add(wt.ka, wsum_dd(dd{kind == 2 && hit < 0 ? wi * Eka : RF(0.0), RF(0.0)}));
        wt.ion = dd_sub(wt.ion, wsum_dd(dd{kind == 1 ? wi * EA : (kind == 2 ? wi * Eka : RF(0.0)), RF(0.0)}));
        __syncwarp();
    }
    if (nb && lane < nb) {
        ph2 *ph = a.photons + S.ph_off + (size_t)c.lc * nb;
        ph2 v = ph[lane];
        dd r = dd_add(dd{v.hi, v.lo}, addph[lane]);
        ph[lane] = ph2{r.hi, r.lo};
    }
    wt.cnt[C_AUG] += wsum_i(c_aug);
    wt.cnt[C_KA] += wsum_i(c_ka);
    __syncwarp();
}

// One cell by its team of TW warps (t of nt = 32 TW threads).  TW = 1: every
// warp of the block takes at most one cell a round, and the stages are
// separated by block barriers so that the warps of an SM fetch the same code
// at the same time (the stages are long and the instruction cache small).
// TW > 1: the block owns one cell.  Per-particle work is spread over the
// team; every sum is formed by one warp over the canonical order (lane-
// strided, fixed tree), so it has the same bits whatever TW is.
template <int TW>
__device__ __forceinline__ void team_sync()
{
    if constexpr (TW == 1) __syncwarp();
    else __syncthreads();
}

template <int RMAX, int TW, bool EARLY>
__device__ void process_cell(const CellArgs &a, const CellMem &m, const Tables &T, int g, int warp, int lane,
                             WarpTally &wt, LaneTally &lt, const int *next)
{
    constexpr int nt = 32 * TW;
    const int t0 = TW == 1 ? lane : warp * 32 + lane;
    // the warps of a team that form its sums (one warp: all of them)
    const bool w0 = TW == 1 || warp == 0, w1 = TW == 1 || warp == 1, w2 = TW == 1 || warp == 2,
               w3 = TW == 1 || warp == 3;
    bool on = g >= 0;
    int s = 0;
    const SlabDev *Sp = a.slabs;
    unsigned step = 0, flags = 0;
    unsigned long long seed = 0;
    int lc = 0, e0 = 0, ne = 0, i0 = 0, ni = 0;
    if (on) {
        s = __ldg(a.cell_slab + g);
        if (s != wt.slab) { tally_flush(a, wt, lt, lane); wt.slab = s; }
        Sp = a.slabs + s;
        step = a.steps[s];
        seed = Sp->seed;
        flags = Sp->flags;
        lc = g - Sp->cell0;
        e0 = a.cs_e[g]; ne = a.cs_e[g + 1] - e0;
        i0 = a.cs_i[g]; ni = a.cs_i[g + 1] - i0;
        on = (ne > 0 || ni > 0) && Sp->active;
    }
    const SlabDev &S = *Sp;
    const real wi = S.w_ion;
    const real mi = S.m_ion;
    const real dt = S.dt;
    const bool rad = S.rad_every > 0 && (step % (unsigned)S.rad_every) == 0;
    const real MC2 = (real)kMeC2;
    const real mw_i = r_mul(r_mul(wi, MC2), mi);      // kinetic energy of an ion per gamma - 1
    const real nref = S.nref_f;
    real n_e = RF(0.), n_i = RF(0.), Te = RF(0.), zbar = RF(0.), lnL = RF(2.);
    const bool coll = (flags & 3u) != 0;
    const real E_bulk = S.E_bulk;
    const bool all_bulk = E_bulk <= RF(0.0);
    dd Kpre = dd_zero();
    int nnew = 0;
    real Wnew_imp = RF(0.0);
    // sums carried from stage to stage (see CellCtx)
    dd Qcell = dd_zero(), Kall = dd_zero(), Kt = dd_zero(), paid_cell = dd_zero();
    real We_cell = RF(0.0);
    int n_imp = 0;
    bool ew_ready = false, ionized = false;

    if (on) {
    // ---- canonical order, then the records staged in it ----
    unsigned *words = reinterpret_cast<unsigned *>(m.ew);
    {
        const RecKeys K{a.e1 + e0, true, seed, step};
        for (int k = t0; k < ne; k += nt) prefetch_l2(a.e0 + e0 + k);
        const unsigned mask = order_cell<RMAX, TW>(K, words, words + ne, ne, warp, lane);
        for (int b0 = 0; b0 < ne; b0 += 2 * nt) {         // two records a thread in flight
            real4 P0[2], P1[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int k = b0 + j * nt + t0;
                if (k >= ne) break;
                const int sl = (int)(words[k] & mask);
                P0[j] = a.e0[e0 + sl];
                P1[j] = a.e1[e0 + sl];
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int k = b0 + j * nt + t0;
                if (k >= ne) break;
                m.eu[k] = make_real4(P0[j].z, P0[j].w, P1[j].x, P1[j].y);
                m.epos[k] = make_real2(P0[j].x, P0[j].y);
                m.eid[k] = rec_eid(P1[j]);
            }
        }
        team_sync<TW>();
    }
    {
        const RecKeys K{a.i1 + i0, false, seed, step};
        const unsigned mask = order_cell<RMAX, TW>(K, words, words + ni, ni, warp, lane);
        for (int k = t0; k < ni; k += nt) {
            const int sl = (int)(words[k] & mask);
            const real4 P0 = a.i0[i0 + sl], P1 = a.i1[i0 + sl];
            m.iu[k] = make_real4(P0.z, P0.w, P1.x, P1.y);
            m.ipos[k] = make_real2(P0.x, P0.y);
            m.ist[k] = rec_ist(P1);
            m.iid[k] = rec_iid(P1);
        }
        team_sync<TW>();
    }
    }

    if (on && rad && S.rt) {
    // ---- transport mode: the energy the radiation field gave up to (or
    //      took from) this cell goes to its bulk electrons by one factor on
    //      their kinetic energy (Sec. II), at most 90 % of it taken; the rest
    //      waits for the next rad step ----
    if (w0) {
    if (lane < S.nb) S.rt_chi[(size_t)lc * S.nb + lane] = 0.0f;
    if (lane == 0) S.rt_emc[lc] = 0.0;
    const double dEc = S.rt_dE[lc];
    if (dEc != 0.0) {
        dd pk = dd_zero();
        for (int k = lane; k < ne; k += 32) {
            const real4 u = m.eu[k];
            const real ke = MC2 * gm1(u.x, u.y, u.z);
            if (E_bulk <= RF(0.0) || ke < E_bulk) pk = dd_addf(pk, u.w * ke);
        }
        const real K = dd_f(wsum_dd(pk));
        if (K > RF(0.0)) {
            const real dEa = (real)dEc < -RF(0.9) * K ? -RF(0.9) * K : (real)dEc;
            const real delta = -dEa / K;
            for (int k = lane; k < ne; k += 32) {
                real4 u = m.eu[k];
                const real ke = MC2 * gm1(u.x, u.y, u.z);
                if (E_bulk <= RF(0.0) || ke < E_bulk) { scale_kinetic(u.x, u.y, u.z, delta); m.eu[k] = u; }
            }
            if (lane == 0) S.rt_dE[lc] = dEc - (double)dEa;
            wt.rt = dd_addf(wt.rt, dEa);
        }
    }
    }
    team_sync<TW>();
    }

    if (on) {
    // ---- cell moments (Sec. II: T_e = 2/3 E_ave over bulk electrons) ----
    // with every electron bulk (the default) the bulk sums are the sums
    dd We = dd_zero(), Wb = dd_zero(), Kb = dd_zero(), Q = dd_zero(), Ka = dd_zero(), Ki = dd_zero();
    if (all_bulk) {
        if constexpr (TW == 1) {
            for (int k = lane; k < ne; k += 32) {
                const real4 u = m.eu[k];
                const real g1 = gm1(u.x, u.y, u.z);
                We = dd_addf(We, u.w);
                Kb = dd_addf(Kb, r_mul(r_mul(u.w, MC2), g1));
            }
        } else {
            if (w0) for (int k = lane; k < ne; k += 32) We = dd_addf(We, m.eu[k].w);
            if (w1)
                for (int k = lane; k < ne; k += 32) {
                    const real4 u = m.eu[k];
                    const real g1 = gm1(u.x, u.y, u.z);
                    Kb = dd_addf(Kb, r_mul(r_mul(u.w, MC2), g1));
                }
        }
    } else if (w0) {
        for (int k = lane; k < ne; k += 32) {
            const real4 u = m.eu[k];
            const real g1 = gm1(u.x, u.y, u.z);
            const real ke = MC2 * g1;
            const real wk = r_mul(r_mul(u.w, MC2), g1);
            We = dd_addf(We, u.w);
            if (ke < E_bulk) { Wb = dd_addf(Wb, u.w); Kb = dd_addf(Kb, wk); }
            Ka = dd_addf(Ka, wk);
        }
    }
    if (w2) for (int k = lane; k < ni; k += 32) Q = dd_addf(Q, (real)(m.ist[k] & 0xff) + m.iu[k].w);
    if (w3 && coll)
        for (int k = lane; k < ni; k += 32) { real4 u = m.iu[k]; Ki = dd_addp(Ki, mw_i, gm1(u.x, u.y, u.z)); }
    if constexpr (TW == 1) {
        wsum_dd4(We, Kb, Q, Ki, lane);
        if (!all_bulk) wsum_dd2(Wb, Ka, lane);
    } else {
        if (w0) {
            We = wsum_dd(We);
            if (lane == 0) m.bc[0] = We;
            if (!all_bulk) {
                Kb = wsum_dd(Kb); Wb = wsum_dd(Wb); Ka = wsum_dd(Ka);
                if (lane == 0) { m.bc[1] = Kb; m.bc[4] = Wb; m.bc[5] = Ka; }
            }
        }
        if (w1 && all_bulk) { Kb = wsum_dd(Kb); if (lane == 0) m.bc[1] = Kb; }
        if (w2) { Q = wsum_dd(Q); if (lane == 0) m.bc[2] = Q; }
        if (w3) { Ki = wsum_dd(Ki); if (lane == 0) m.bc[3] = Ki; }
        __syncthreads();
        We = m.bc[0]; Kb = m.bc[1]; Q = m.bc[2]; Ki = m.bc[3];
        if (!all_bulk) { Wb = m.bc[4]; Ka = m.bc[5]; }
    }
    if (all_bulk) { Wb = We; Ka = Kb; }
    Kall = Ka;
    Qcell = Q;
    We_cell = dd_f(We);
    n_e = dd_f(We) * nref; n_i = (real)ni * wi * nref;
    Te = dd_f(Wb) > RF(0.0) ? (RF(2.0) / RF(3.0)) * dd_f(Kb) / dd_f(Wb) : RF(0.0);
    zbar = ni > 0 ? dd_f(Q) / ni : RF(0.0);
    if (w0 && lane < NZ) m.dE[lane] = ipd_shift(S.ipd, lane, n_e, n_i, Te, zbar);
    lnL = S.coulomb_log > RF(0.0) ? S.coulomb_log : coulomb_log(n_e, Te, zbar);
    if constexpr (TW == 1) __syncwarp();

    // ---- binary collisions (Sec. IV): e-e, then e-i; exact energy restore ----
    if (coll) Kpre = dd_add(Kall, Ki);
    if ((flags & 1u) && ne >= 2) {
        auto ee = [&](int pa, int pb, real dtc) {
            const real4 A = m.eu[pa], B = m.eu[pb];
            const U4 r = draw(seed, m.eid[pa], step, PU_COLL_EE);
            const Collided q = binary_collision(A, B, RF(1.0), RF(1.0), -RF(1.0), -RF(1.0), A.w, B.w, n_e, lnL, dtc, coll_draw(r));
            lt.ee += q.hit;
            m.eu[pa] = q.a;
            m.eu[pb] = q.b;
        };
        // an odd count pairs its first three in a triangle at half the step
        const int start = (ne & 1) ? 3 : 0;
        const int npairs = (ne - start) >> 1;
        if (start && t0 == 0)
#pragma unroll 1
            for (int q = 0; q < 3; ++q) ee(q, q == 2 ? 0 : q + 1, RF(0.5) * dt);
#pragma unroll 1
        for (int p = t0; p < npairs; p += nt) ee(start + 2 * p, start + 2 * p + 1, dt);
    }
    team_sync<TW>();
    }
    // the cell this warp takes next: where its records are, for a prefetch
    // into L2 after this cell's e-i collisions
    [[maybe_unused]] int pe0 = 0, pe1 = 0, pi0 = 0, pi1 = 0;
    if constexpr (TW == 1) __syncthreads();     // the e-i code next: warps in step, as elsewhere
    if constexpr (EARLY) {
        const int gn = *next + warp;
        if (gn < a.ncell) { pe0 = a.cs_e[gn]; pe1 = a.cs_e[gn + 1]; pi0 = a.cs_i[gn]; pi1 = a.cs_i[gn + 1]; }
    }

    if (on) {
    if ((flags & 2u) && ne >= 1 && ni >= 1) {
        // the longer species in order, the shorter cycled: particle t of the
        // shorter meets t, t + nshort, ... of the longer, one after another,
        // and no other thread touches any of them
        if (ne >= ni) {
            // The chains keep as many lanes busy as there are ions (16 to 20
            // of 32 in the 2D workloads); the draws, half of a collision's
            // instructions, depend on the electron alone, so one warp forms
            // them first with all its lanes.
            constexpr bool STAGED = RMAX <= 128 && TW == 1;
            if constexpr (STAGED) {
                for (int pe = lane; pe < ne; pe += 32) {
                    const CollDraw d = coll_draw(draw(seed, m.eid[pe], step, PU_COLL_EI));
                    m.rn[pe] = make_real4(d.a, d.c, d.sphi, d.cphi);
                    m.ew[pe].x = d.r3;
                }
                __syncwarp();
            }
            for (int pi = t0; pi < ni; pi += nt) {
                real4 B = m.iu[pi];
                const real q = (real)(m.ist[pi] & 0xff) + B.w;
#pragma unroll 1
                for (int pe = pi; pe < ne; pe += ni) {
                    const real4 A = m.eu[pe];
                    const real npair = n_i * r_fmax(A.w, wi) / wi;
                    CollDraw d;
                    if constexpr (STAGED) {
                        const real4 v = m.rn[pe];
                        d = CollDraw{v.x, v.y, v.z, v.w, m.ew[pe].x};
                    } else {
                        d = coll_draw(draw(seed, m.eid[pe], step, PU_COLL_EI));
                    }
                    const Collided c = binary_collision(A, B, RF(1.0), mi, -RF(1.0), q, A.w, wi, npair, lnL, dt, d);
                    lt.ei += c.hit;
                    m.eu[pe] = c.a;
                    B = c.b;
                }
                m.iu[pi] = B;
            }
        } else {
            for (int pe = t0; pe < ne; pe += nt) {
                real4 A = m.eu[pe];
#pragma unroll 1
                for (int pi = pe; pi < ni; pi += ne) {
                    const real4 B = m.iu[pi];
                    const real q = (real)(m.ist[pi] & 0xff) + B.w;
                    const real npair = n_e * r_fmax(A.w, wi) / A.w;
                    const U4 r = draw(seed, (unsigned long long)m.iid[pi], step, PU_COLL_IE);
                    const Collided c = binary_collision(A, B, RF(1.0), mi, -RF(1.0), q, A.w, wi, npair, lnL, dt, coll_draw(r));
                    lt.ei += c.hit;
                    A = c.a;
                    m.iu[pi] = c.b;
                }
                m.eu[pe] = A;
            }
        }
        team_sync<TW>();
    }
    if (coll && ne >= 1) {
        // kinetic energies after the collisions; each electron's gamma - 1
        // stays in the scratch for the passes below
        dd Ke = dd_zero(), Ki = dd_zero();
        if constexpr (TW == 1) {
            for (int k = lane; k < ne; k += 32) {
                const real4 u = m.eu[k];
                const real g1 = gm1(u.x, u.y, u.z);
                m.ew[k].x = g1;
                Ke = dd_addp(Ke, r_mul(u.w, MC2), g1);
            }
            for (int k = lane; k < ni; k += 32) { real4 u = m.iu[k]; Ki = dd_addp(Ki, mw_i, gm1(u.x, u.y, u.z)); }
            wsum_dd2(Ke, Ki, lane);
        } else {
            for (int k = t0; k < ne; k += nt) { const real4 u = m.eu[k]; m.ew[k].x = gm1(u.x, u.y, u.z); }
            __syncthreads();
            if (w0) {
                for (int k = lane; k < ne; k += 32) Ke = dd_addp(Ke, r_mul(m.eu[k].w, MC2), m.ew[k].x);
                Ke = wsum_dd(Ke);
                if (lane == 0) m.bc[0] = Ke;
            }
            if (w1) {
                for (int k = lane; k < ni; k += 32) { real4 u = m.iu[k]; Ki = dd_addp(Ki, mw_i, gm1(u.x, u.y, u.z)); }
                Ki = wsum_dd(Ki);
                if (lane == 0) m.bc[1] = Ki;
            }
            __syncthreads();
            Ke = m.bc[0]; Ki = m.bc[1];
        }
        real ke = dd_f(Ke);
        real delta = RF(0.0);
        if (ke > RF(0.0)) {
            delta = -dd_f(dd_sub(dd_sub(Kpre, Ke), Ki)) / ke;     // f = 1 - delta
            if (!(delta < RF(1.0))) delta = RF(0.0);
        }
        if ((flags & 4u) && ni >= 1) {
            // the restore and the ionization stage's per-electron inputs in
            // one pass: kinetic energy and w * beta after the restore, and
            // the kinetic energies' sum
            dd pt = dd_zero();
            for (int k = t0; k < ne; k += nt) {
                real4 u = m.eu[k];
                scale_kinetic(u.x, u.y, u.z, m.ew[k].x, delta);
                m.eu[k] = u;
                real u2 = square3_yx(u.x, u.y, u.z);
                real g1 = gm1_of(u2);
                if constexpr (TW == 1) pt = dd_addp(pt, r_mul(u.w, MC2), g1);
                m.ew[k] = make_real2(MC2 * g1, u.w * (r_sqrt(u2) / (RF(1.0) + g1)));
            }
            if constexpr (TW == 1) Kt = wsum_dd(pt);
            ew_ready = true;
        } else if (delta != RF(0.0)) {
            for (int k = t0; k < ne; k += nt) {
                real4 u = m.eu[k];
                scale_kinetic(u.x, u.y, u.z, m.ew[k].x, delta);
                m.eu[k] = u;
            }
        }
        team_sync<TW>();
    }

    }
    if constexpr (TW == 1) __syncthreads();
    if constexpr (EARLY) {
        constexpr int PER = 128 / sizeof(real4);
        const bool elec = lane < 24;
        const int k = (elec ? pe0 : pi0) + PER * (elec ? lane % 12 : lane % 4);
        if (k < (elec ? pe1 : pi1)) prefetch_l2((elec ? (lane < 12 ? a.e0 : a.e1) : (lane < 28 ? a.i0 : a.i1)) + k);
    }

    if (on) {
    // ---- Lotz impact ionization, cell-average probability (Eq. 3) ----
    if ((flags & 4u) && ne >= 1 && ni >= 1) {
        // charge states present (every warp of a team for itself)
        unsigned pmask = 0;
        for (int k = lane; k < ni; k += 32) { int Z = m.ist[k] & 0xff; if (Z < ZNUC) pmask |= 1u << Z; }
        pmask = __reduce_or_sync(FULL, pmask);
        // kinetic energy and w * beta of each electron (canonical order)
        real2 *ew = m.ew;
        int nhot = 0;
        if (!ew_ready) {
            dd pk = dd_zero();
            for (int k = t0; k < ne; k += nt) {
                real4 u = m.eu[k];
                real u2 = square3(u.x, u.y, u.z);
                real g1 = gm1_of(u2);
                if constexpr (TW == 1) pk = dd_addp(pk, r_mul(u.w, MC2), g1);
                ew[k] = make_real2(MC2 * g1, u.w * (r_sqrt(u2) / (RF(1.0) + g1)));
            }
            if constexpr (TW == 1) Kt = wsum_dd(pk);
            team_sync<TW>();
        }
        // Electrons at or below the lowest lowered binding of every charge
        // state present ionize nothing and add nothing to the sums: the
        // others (a hot tail, typically a few per cent) are gathered in
        // canonical order to the front of the storage, so that a warp's
        // lanes do not idle beside the one lane with a hot electron.
        if (TW > 1 && w1) {
            dd pt = dd_zero();
            for (int k = lane; k < ne; k += 32) {
                const real4 u = m.eu[k];
                real u2 = ew_ready ? square3_yx(u.x, u.y, u.z) : square3(u.x, u.y, u.z);
                real g1 = gm1_of(u2);
                pt = dd_addp(pt, r_mul(u.w, MC2), g1);
            }
            pt = wsum_dd(pt);
            if (lane == 0) m.bc[2] = pt;
        }
        if (w0) {
            real Pall = RF(3.0e38);
            for (int z = 0; z < ZNUC; ++z) {
                if (!(pmask & (1u << z))) continue;
                if (lane < NS && subshell_occ(ZNUC - z, lane) > 0)
                    Pall = r_fmin(Pall, lowered_binding(T, z, lane, m.dE[z]));
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) Pall = r_fmin(Pall, __shfl_xor_sync(FULL, Pall, o));
            Pall = __shfl_sync(FULL, Pall, 0);
            int nh = 0;
            for (int b0 = 0; b0 < ne; b0 += 32) {
                const int k = b0 + lane;
                const real2 q = k < ne ? ew[k] : make_real2(RF(0.0), RF(0.0));
                const bool hot = k < ne && q.x > Pall;
                const unsigned bal = __ballot_sync(FULL, hot);
                __syncwarp();
                if (hot) ew[nh + __popc(bal & ((1u << lane) - 1u))] = q;
                nh += __popc(bal);
                __syncwarp();
            }
            nhot = nh;
            if (TW > 1 && lane == 0) m.bc[3].hi = (real)nh;
        }
        if constexpr (TW > 1) {
            __syncthreads();
            Kt = m.bc[2];
            nhot = (int)m.bc[3].hi;
        }
        // Charge states side by side: with a few hot electrons the lanes form
        // groups of 8, 16 or 32, a charge state each (what the lanes beyond
        // nhot would add to a sum's tree is zero).
        const real cfac = (real)(kCcmPerFs) * dt * nref;
        real4 *lz = m.lz + (TW == 1 ? 0 : warp * LOTZ_SETS * NS);
        const int G = nhot <= 8 ? 8 : (nhot <= 16 ? 16 : 32), gl = lane & (G - 1), gi = lane / G, per = 32 / G;
        unsigned zs = pmask;                         // charge states to come
        auto drop = [](unsigned v, int n) { for (int j = 0; j < n; ++j) v &= v - 1u; return v; };
        if (TW > 1) zs = drop(zs, warp * per);
        for (; zs; zs = drop(zs, TW * per)) {
            // the group's charge state: the gi-th of them (-1: none)
            const int z = __ffs(drop(zs, gi)) - 1;
            // Lotz constants of charge state z (lowest-energy configuration):
            // lowered binding P, 1/P, ln P, a * occupation (0: empty subshell)
            if (gl < NS) {
                const int o = z >= 0 ? subshell_occ(ZNUC - z, gl) : 0;
                real4 v = make_real4(RF(0.0), RF(0.0), RF(0.0), RF(0.0));
                if (o > 0) {
                    const real P = lowered_binding(T, z, gl, m.dE[z]);
                    v = make_real4(P, RF(1.0) / P, r_log(P), T.lotz_a[gl] * (real)o);
                }
                lz[gi * NS + gl] = v;
            }
            __syncwarp();
            // fast log / exp: a few ulp on a probability; only a decision
            // within that of its threshold could flip
            dd pr = dd_zero();
            for (int k = gl; k < nhot; k += G) {
                const real2 q = ew[k];
                const real E = q.x, lnE = r_flog(E), invE = RF(1.0) / E;
                real sig = RF(0.0);
                bool any = false;
#pragma unroll
                for (int sh = 0; sh < NS; ++sh) {
                    const real4 L = lz[gi * NS + sh];
                    if (L.w > RF(0.0) && E > L.x) {
                        const real x = E * L.y;
                        sig += L.w * (lnE - L.z) * (invE * L.y) *
                               (RF(1.0) - T.lotz_b[sh] * r_fexp(-T.lotz_c[sh] * (x - RF(1.0))));
                        any = true;
                    }
                }
                // at or below the lowest binding of the charge state: nothing
                if (any) pr = dd_addp(pr, q.y, sig);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (o < G) {
                    dd t{__shfl_xor_sync(FULL, pr.hi, o), __shfl_xor_sync(FULL, pr.lo, o)};
                    pr = dd_add(pr, t);
                }
            const real P = cfac * dd_f(pr);
            if (gl == 0 && z >= 0) m.Pz[z] = P;
            wt.cnt[C_PGT1] += __popc(__ballot_sync(FULL, gl == 0 && z >= 0 && P > RF(1.0)));
            __syncwarp();
        }
        team_sync<TW>();
        dd paid = dd_zero();
        if (w0) {
            dd carry = dd_zero();
            for (int b0 = 0; b0 < ni; b0 += 32) {
                int t = b0 + lane;
                bool cand = false;
                real cost = RF(0.0);
                int Z = 0, nK = 0;
                if (t < ni) {
                    int st = m.ist[t];
                    Z = st & 0xff; nK = (st >> 8) & 0xff;
                    if (Z < ZNUC) {
                        U4 r = draw(seed, (unsigned long long)m.iid[t], step, PU_ION);
                        if (u01(r.x) < m.Pz[Z]) {
                            cand = true;
                            cost = wi * removal_energy(T, Z, nK, m.dE[Z]);
                        }
                    }
                }
                // no candidate among these ions (most cells): nothing to pay
                if (!__any_sync(FULL, cand)) continue;
                dd incl = dd_add(carry, wscan_dd(dd{cost, RF(0.0)}, lane));
                bool acc = cand && dd_le(incl, Kt);
                if (cand && !acc) lt.rej++;
                unsigned bal = __ballot_sync(FULL, acc);
                if (acc) {
                    int so = outer_shell(ZNUC - Z, nK);
                    lose_electron(Z, nK, so);
                    m.ist[t] = Z | (nK << 8);
                    int pos = nnew + __popc(bal & ((1u << lane) - 1u));
                    if (pos < a.cap_new) {
                        NewE q; q.ux = q.uy = q.uz = RF(0.0); q.w = wi; q.meta = t | (KIND_IMPACT << 16);
                        m.nw[pos] = q;
                    } else {
                        atomicOr(a.err, ERR_NEW_OVERFLOW);
                    }
                    lt.ion++;
                }
                paid = dd_add(paid, wsum_dd(dd{acc ? cost : RF(0.0), RF(0.0)}));
                nnew += __popc(bal);
                n_imp += __popc(bal);
                carry = wlane_dd(incl, 31);
            }
            nnew = min(nnew, a.cap_new);
            if (TW > 1 && lane == 0) m.bc[4] = paid;
        }
        if constexpr (TW > 1) {
            __syncthreads();
            paid = m.bc[4];
        }
        Wnew_imp = nnew * wi;
        paid_cell = paid;
        ionized = true;
        real pf = dd_f(paid);
        if (pf > RF(0.0)) {
            real delta = pf / dd_f(Kt);
            for (int k = t0; k < ne; k += nt) {
                real4 u = m.eu[k];
                scale_kinetic(u.x, u.y, u.z, gm1(u.x, u.y, u.z), delta);
                m.eu[k] = u;
            }
            if (w0) wt.ion = dd_add(wt.ion, paid);
        }
        team_sync<TW>();
    }

    }
    if constexpr (TW == 1) __syncthreads();

    if (on) {
    if ((flags & 8u) && ni >= 1) {
        CellCtx cc;                       // (inline: in registers)
        cc.ne = ne; cc.ni = ni; cc.n_i = n_i;
        cc.have_sums = all_bulk && ionized;
        cc.K_after = dd_sub(Kt, paid_cell);
        cc.W_e = We_cell;
        cc.Q_after = dd_f(Qcell) + (real)n_imp;
        real delta = RF(0.0);
        bool rec = false;
        if (w0) {
            real Wex;
            const int Kev = recombine_wanted(a, m, E_bulk, cc, lane, Wnew_imp, Wex);
            if (Kev > 0) rec = stage_recombine(a, m, T, E_bulk, wi, ne, ni, lane, Kev, Wex, wt, delta);
            if (TW > 1 && lane == 0) m.bc[5] = dd{delta, rec ? RF(1.0) : RF(0.0)};
        }
        if constexpr (TW > 1) {
            __syncthreads();
            delta = m.bc[5].hi;
            rec = m.bc[5].lo != RF(0.0);
        }
        if (rec) recombine_apply(m, S, ne, delta, t0, nt);
        team_sync<TW>();
    }
    if (rad && w0) {
        CellCtx cc;
        cc.lc = lc; cc.ne = ne; cc.ni = ni;
        cc.step = step; cc.seed = seed; cc.wi = wi; cc.n_i = n_i; cc.nref = nref;
        if ((flags & 16u) && S.nb && ni >= 1) stage_photo(a, m, T, S, cc, lane, nnew, wt);
        if ((flags & 32u) && ni >= 1) stage_decay(a, m, T, S, cc, lane, nnew, wt);
        if (flags & 256u) stage_therm(m, cc, lane, nnew);
    }
    if (TW > 1 && rad) __syncthreads();

    // ---- write the collided state back, each cell's records in its
    //      canonical order (the order the push kernel follows) ----
    for (int k = t0; k < ne; k += nt) {
        const real4 u = m.eu[k];
        const real2 x = m.epos[k];
        a.e0[e0 + k] = make_real4(x.x, x.y, u.x, u.y);
        a.e1[e0 + k] = rec_e1(u.z, u.w, m.eid[k]);
    }
    for (int k = t0; k < ni; k += nt) {
        const real4 u = m.iu[k];
        const real2 x = m.ipos[k];
        a.i0[i0 + k] = make_real4(x.x, x.y, u.x, u.y);
        a.i1[i0 + k] = rec_i1(u.z, u.w, m.iid[k], m.ist[k]);
    }
    if (rad && S.rt && w0) {
        // transport mode: the cell's electron weight after the step, created
        // electrons included: its share of the next heating of its rad cell
        // (summed in canonical order: the slots' order is the scatter's)
        real wsum = RF(0.0);
        for (int k = lane; k < ne; k += 32) {
            const real w = m.eu[k].w;
            wsum += w > RF(0.0) ? w : RF(0.0);
        }
        for (int k = lane; k < nnew; k += 32) wsum += m.nw[k].w;
        wsum = wsum_f(wsum);
        if (lane == 0) S.rt_w[lc] = (float)wsum;
    }
    // ---- created electrons: after the sorted range, at their ion, with their cell as key ----
    if (w0 && nnew > 0) {
        // a slab with a budget of its own keeps its electrons within it: a
        // cell that would take it beyond drops what it created and fails
        // the slab alone (it is stopped at the end of the step); the others
        // never see the shared capacity run out when the budgets fit in it
        int base = 0, fits = 1;
        if (lane == 0) {
            if (S.budget_e > 0) {
                const int held = a.cs_e[S.cell0 + S.ncell] - a.cs_e[S.cell0];
                if (held + atomicAdd(a.slab_app + s, nnew) + nnew > S.budget_e) {
                    atomicOr(a.slab_err + s, ERR_CAPACITY);
                    fits = 0;
                }
            }
            if (fits) base = atomicAdd(a.append, nnew);
        }
        fits = __shfl_sync(FULL, fits, 0);
        base = __shfl_sync(FULL, base, 0);
        const int sorted = a.cs_e[a.ncell];
        int n_ok = fits ? nnew : 0;
        if (fits && sorted + base + nnew > a.cap_e) {
            if (lane == 0) atomicOr(a.err, ERR_CAPACITY);
            for (int k = sorted + base + lane; k < min(a.cap_e, sorted + base + nnew); k += 32) a.ekey[k] = -1;
            n_ok = 0;
        }
        for (int k = lane; k < n_ok; k += 32) {
            NewE q = m.nw[k];
            const int ip = q.meta & 0xffff, kind = q.meta >> 16;
            const real2 x = m.ipos[ip];
            unsigned idhi = ((step + 1u) << 2) | (unsigned)kind;
            a.e0[sorted + base + k] = make_real4(x.x, x.y, q.ux, q.uy);
            a.e1[sorted + base + k] = rec_e1(q.uz, q.w, ((unsigned long long)idhi << 32) | m.iid[ip]);
            a.ekey[sorted + base + k] = g;
        }
    }
    }
    __syncthreads();
}

// Bound by instruction issue and the latency of dependent chains at 16
// resident warps per SM (128 registers); its memory side moves only the 64 B
// per particle.  So it is written for few instructions per particle: the
// order sorts 32-bit words, the records are staged in that order (no index
// loads, no bank conflicts), up to four cell sums share one reduction, each
// electron's gamma - 1 is kept between the collision restore's two passes,
// the collisions are inline with their particles in registers, and an ion
// keeps its state in registers through its chain of collisions.  Against the
// 64-bit sort, slot-ordered staging, one reduction per sum and collisions
// called by reference: 2048 x 256 cells of 64 e + 16 i, 42 M particles, 6.94
// -> 5.40 ms a step; 512 x 64 cells 511 -> 397 us.  With the Lotz sums of
// several charge states side by side, the recombination clamp inline, the
// e-i draws formed ahead of their chains and the next cell's records
// prefetched: 4.88 ms and 364 us.  Two CTAs of 8 warps an SM: 6 to 10 warps a
// CTA at 80 to 112 registers (18 to 24 warps an SM) take 5.2 to 6.0 ms, one
// CTA of 16 warps 5.4.
// Each round the block takes one cell per team from a shared counter.
// Cells whose population exceeds this launch's shared-memory capacity go to
// a list for the next launch.
// RMAX: the most entries per species a launch stages; TW: warps per cell.
// EARLY: a block takes its next round's cells while it computes this one's
// and prefetches their records into L2; for launches of many rounds over all
// cells (with few rounds, a block that took its cells early leaves them
// waiting while others are idle).
template <int RMAX, int TW, bool EARLY = false>
__global__ void __launch_bounds__(TW == 1 ? 256 : 32 * TW, TW == 1 ? 2 : 16 / TW) k_cell(CellArgs a)
{
    extern __shared__ __align__(kSmAlign) char smem[];
    __shared__ Tables T;
    __shared__ int s_next;               // first cell of the block's next round
    const int total = a.list ? *a.n_list : a.ncell;
    if (total == 0) return;              // a tier no cell needs
    for (int k = threadIdx.x; k < (int)(sizeof(Tables) / sizeof(real)); k += blockDim.x)
        ((real *)&T)[k] = ((const real *)a.tab)[k];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nteam = TW == 1 ? blockDim.x >> 5 : 1;
    const int team = TW == 1 ? warp : 0;
    CellMem m = carve(smem + (size_t)team * cell_mem_bytes(a.cap_ce, a.cap_ci, TW), a.cap_ce, a.cap_ci, TW,
                      a.nw + ((size_t)blockIdx.x * nteam + team) * a.cap_new);
    WarpTally wt;
    LaneTally lt{0, 0, 0, 0};
    wt.slab = -1;
    wt.ion = wt.ka = wt.esc = wt.rt = dd_zero();
    for (int q = 0; q < NCOUNT; ++q) wt.cnt[q] = 0;
    if (EARLY && threadIdx.x == 0) s_next = atomicAdd(a.work, nteam);
    for (;;) {
        __syncthreads();
        if (!EARLY && threadIdx.x == 0) s_next = atomicAdd(a.work, nteam);
        if (!EARLY) __syncthreads();
        const int base = s_next;
        if (base >= total) break;
        if (EARLY) {
            __syncthreads();
            if (threadIdx.x == 0) s_next = atomicAdd(a.work, nteam);
        }
        int g = -1;
        if (base + team < total) {
            g = a.list ? a.list[base + team] : base + team;
            int ne = a.cs_e[g + 1] - a.cs_e[g], ni = a.cs_i[g + 1] - a.cs_i[g];
            if (ne > a.cap_ce || ni > a.cap_ci || 3 * ni > a.cap_new) {
                if (TW == 1 || warp == 0) {
                    if (a.ovf_list) {
                        if (lane == 0) a.ovf_list[atomicAdd(a.ovf_count, 1)] = g;
                    } else {
                        // no larger pass left: report, and drop the cell's particles so
                        // that the next sort stays consistent
                        if (lane == 0) atomicOr(a.err, ERR_CELL_OVERFLOW);
                        for (int k = a.cs_e[g] + lane; k < a.cs_e[g + 1]; k += 32)
                            reinterpret_cast<real *>(a.e1 + k)[1] = RF(0.0);
                        for (int k = a.cs_i[g] + lane; k < a.cs_i[g + 1]; k += 32) a.i1[k].w = bits_real(0xffu);
                    }
                }
                g = -1;
            }
        }
        process_cell<RMAX, TW, EARLY>(a, m, T, g, warp, lane, wt, lt, &s_next);
    }
    tally_flush(a, wt, lt, lane);
}

}  // namespace pic
