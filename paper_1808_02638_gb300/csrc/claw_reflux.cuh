// claw_reflux.cuh -- the conservation fix of Sec. 2.3 ("refluxing") for a uniform medium, where
// the acoustics system is in conservation form: f(Q) = A Q, g(Q) = B Q, and for the shallow water
// equations, whose Roe solver is conservative (A-dQ + A+dQ = f(Q_R) - f(Q_L)): there A (Q_F - Q_C)
// below becomes f(Q_F) - f(Q_C) with the equations' own flux.
//
// A coarse cell C next to the fine region (not covered by it) is updated by the coarse step with
// the flux F_e through its edge e; the fine cells along e see r fine fluxes per substep.  After
// the fine substeps and the average, C is corrected so that the flux through e is the average
// of the fine ones.  With C left of e and fine cells F_b right of their edges e_b:
//   F_e   - f(Q_C^n) = A-dQ_e + F~_e                                  (coarse part)
//   F_b^k - f(Q_C^n) = A (Q_F^k - Q_C^n) - A+dQ_b^k + F~_b^k            (fine part, substep k)
//   Q_C^{n+1} += -(dt/dx) [ (1/r^2) sum_{k,b} (F_b^k - f(Q_C^n)) - (F_e - f(Q_C^n)) ]
// (the paper's C1 + C2 + C3), mirrored for C right of e (+A-dQ_b, -A+dQ_e, opposite sign) and
// in y.  F~ is the correction flux plus the transverse terms the other direction's sweep puts
// on the edge.  Each edge's quantities are evaluated here from the state the step read, with the
// step's own formulation (wave strengths scaled by 2, the same limiter functions), so the fix
// matches the fused kernel's update to rounding.
//
// Eight lanes evaluate an edge: its quantities need the limited waves of five edges (its own, and the
// two transverse edges of the cell on either side), each from a row of four cells; lane k evaluates
// edge k, all with the same code, and the first combines them.  One thread per edge took a chain of
// some 150 FP64 instructions (12 us a launch with van Leer's reciprocals).
#pragma once

#include "claw_step.cuh"

namespace claw {
namespace refl {

constexpr int kLanes = 8;   // per edge (five work)

// value of lane `from` of the caller's group of eight
__device__ __forceinline__ double lane_of(double x, int from)
{
    return __shfl_sync(0xffffffffu, x, (threadIdx.x & 24) + from);
}

// Five edges of the edge between normal indices e-1 and e on line t (dir 0: x-edge, normal index i,
// line j; dir 1: y-edge): lane 0 itself, lanes 1, 2 the transverse edges t, t+1 at normal index e-1,
// lanes 3, 4 at e.  Cell k (0..3) of this lane's row: the two either side of its edge are 1 and 2.
struct Row {
    const double* q;
    long long o;      // plane-0 element of cell 0
    long long step;   // to the next cell of the row
    long long WH;
    int nm, tm;       // component along the row, across it
    __device__ __forceinline__ Row(const double* base, int W, long long plane, int dir, int e, int t, int lane)
    {
        q = base;
        WH = plane;
        const bool along = lane == 0 || lane > 4;
        const int n = along ? e - 2 : lane < 3 ? e - 1 : e;                 // normal index of cell 0
        const int l = along ? t : (lane == 1 || lane == 3 ? t - 2 : t - 1);   // its line
        const int i = dir == 0 ? n : l, j = dir == 0 ? l : n;
        o = (long long)(j + 2) * W + (i + 2);
        step = (dir == 0) == along ? 1 : W;
        const int mn = dir == 0 ? 1 : 2;
        nm = along ? mn : 3 - mn;
        tm = 3 - nm;
    }
    __device__ __forceinline__ double at(int m, int k) const { return q[m * WH + o + k * step]; }
};

// A-dQ, A+dQ and F~ of an edge, components in its order (p, normal velocity, transverse velocity); valid
// in lane 0
template <int LIM>
__device__ __forceinline__ void edge_terms(const Row& row, int lane, const StepArgs& A, double ln, double lt,
                                           double am[3], double ap[3], double f[3])
{
    const double c = A.c0, Z = A.Z0, iZ = A.iZ;
    double p[4], u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        p[k] = row.at(0, k);
        u[k] = row.at(row.nm, k);
    }
    double x1[3], x2[3];   // strengths (x2) of the edges between cells k, k + 1
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double dp = p[k + 1] - p[k], du = u[k + 1] - u[k];
        x1[k] = fma(-dp, iZ, du);
        x2[k] = fma(dp, iZ, du);
    }
    const bool second = A.order == 2, cw = A.transverse == 2 && second;
    double m1 = 0.0, m2 = 0.0;
    if (second) {
        m1 = Lim<LIM>::f(x1[1], x1[2]);
        m2 = Lim<LIM>::f(x2[1], x2[0]);
    }
    const double a1 = x1[1], a2 = x2[1];
    am[0] = 0.5 * c * Z * a1;
    am[1] = -0.5 * c * a1;
    am[2] = 0.0;
    ap[0] = 0.5 * c * Z * a2;
    ap[1] = 0.5 * c * a2;
    ap[2] = 0.0;
    f[0] = f[1] = f[2] = 0.0;
    if (second) {   // normal correction flux: (1/2) sum |s| (1 - ln |s|) W~
        const double kap = c * (1.0 - ln * c);
        f[0] += 0.25 * kap * Z * (m2 - m1);
        f[1] += 0.25 * kap * (m1 + m2);
    }
    if (A.transverse) {
        // pressure of the transverse fluctuations into a cell: the up-going part of its lower
        // transverse edge (with -C) and the down-going part of the upper one (with +C); lanes 1 and 3
        const double s = m2 - m1;
        const double hi1 = __shfl_down_sync(0xffffffffu, a1, 1), shi = __shfl_down_sync(0xffffffffu, s, 1);
        double r = 0.5 * c * Z * (a2 + hi1);
        if (cw) r += 0.5 * c * (1.0 - lt * c) * Z * (shi - s);
        const double PL = lane_of(r, 1), PR = lane_of(r, 3);
        f[0] -= 0.25 * lt * c * (PL - PR);
        f[1] -= 0.25 * lt * c * iZ * (PL + PR);
    }
}

// ------------------------------------------------------------------ shallow water
// Roe state and wave strengths of one edge: the step kernel's to rounding (per-cell sqrt(h) and momenta over
// sqrt(h), one reciprocal square root for c and 1/(2c); here the reciprocal is a division's and the
// third strength comes from its own speed)
struct SEdge {
    double un, ut, c, i2c, a1, a2, a3;
};

__device__ __forceinline__ SEdge swe_solve(double hl, double nl, double tl, double hr, double nr, double tr, double hg)
{
    const double rl = rsqrt(hl), rr = rsqrt(hr);
    const double inv = 1.0 / (hl * rl + hr * rr);
    SEdge E;
    E.un = (nl * rl + nr * rr) * inv;
    E.ut = (tl * rl + tr * rr) * inv;
    const double x = (hl + hr) * hg;
    const double rc = rsqrt(x);
    E.c = x * rc;
    E.i2c = 0.5 * rc;
    const double dh = hr - hl, dn = nr - nl, dt = tr - tl;
    E.a1 = fma(E.un + E.c, dh, -dn) * E.i2c;
    E.a2 = fma(-E.ut, dh, dt);
    E.a3 = fma(-(E.un - E.c), dh, dn) * E.i2c;
    return E;
}

// h_p = |s_p| (1 - l |s_p|) mu_p / 2 of an edge from itself and its two neighbours along the sweep
template <int LIM>
__device__ __forceinline__ void swe_limited(const SEdge& E, const SEdge& Eb, const SEdge& Ef, double l, double h[3])
{
    const double s1 = E.un - E.c, s3 = E.un + E.c;
    const SEdge& U1 = s1 > 0.0 ? Eb : Ef;
    const SEdge& U2 = E.un > 0.0 ? Eb : Ef;
    const SEdge& U3 = s3 > 0.0 ? Eb : Ef;
    const double w = fma(E.ut, E.ut, 1.0);
    const double rr1 = fma(s1, s1, w), rr3 = fma(s3, s3, w);
    const double ip = 1.0 / (rr1 * rr3);
    const double ri1 = fma(U1.un - U1.c, s1, fma(U1.ut, E.ut, 1.0));
    const double ri3 = fma(U3.un + U3.c, s3, fma(U3.ut, E.ut, 1.0));
    const double mu1 = Lim<LIM>::f(E.a1, U1.a1 * ri1 * (rr3 * ip));
    const double mu2 = Lim<LIM>::f(E.a2, U2.a2);
    const double mu3 = Lim<LIM>::f(E.a3, U3.a3 * ri3 * (rr1 * ip));
    const double k1 = fabs(s1), k2 = fabs(E.un), k3 = fabs(s3), hl = -0.5 * l;
    h[0] = fma(hl * k1, k1, 0.5 * k1) * mu1;
    h[1] = fma(hl * k2, k2, 0.5 * k2) * mu2;
    h[2] = fma(hl * k3, k3, 0.5 * k3) * mu3;
}

// the fluctuation an edge sends into the cell on its right (right) or left, with the correction
// at the weight the transverse mode gives (hw = +1: full C, -1: none), split across the sweep:
// adds the part going to lower transverse indices to bm and the rest to bp, (h, n, t) order
__device__ __forceinline__ void swe_side_split(const SEdge& E, const double h[3], bool right, double hw,
                                               double bm[3], double bp[3])
{
    const double s[3] = {E.un - E.c, E.un, E.un + E.c};
    const double a[3] = {E.a1, E.a2, E.a3};
    double d[3];
    for (int p = 0; p < 3; ++p) {
        const double hp = right ? -h[p] : h[p];
        const double lam = right ? (s[p] > 0.0 ? s[p] : 0.0) : (s[p] < 0.0 ? s[p] : 0.0);
        d[p] = fma(hw, hp, fma(lam, a[p], hp));
    }
    const double dh = d[0] + d[2], t = d[1] * E.i2c;
    const double b[3] = {fma(0.5, dh, -t), E.c * (d[2] - d[0]), fma(0.5, dh, t)};
    const double m[3] = {E.ut - E.c, E.ut, E.ut + E.c};
    double gm[3], gp[3];
    for (int q = 0; q < 3; ++q) {
        const double g = m[q] * b[q];
        gm[q] = m[q] < 0.0 ? g : 0.0;
        gp[q] = m[q] < 0.0 ? 0.0 : g;
    }
    const double Gm = gm[0] + gm[2], Gp = gp[0] + gp[2];
    bm[0] += Gm;
    bm[1] += fma(E.un, Gm, gm[1]);
    bm[2] += fma(E.ut, Gm, E.c * (gm[2] - gm[0]));
    bp[0] += Gp;
    bp[1] += fma(E.un, Gp, gp[1]);
    bp[2] += fma(E.ut, Gp, E.c * (gp[2] - gp[0]));
}

// A-dQ, A+dQ and F~ (correction plus the other sweep's transverse terms) of an edge, components (h,
// normal momentum, transverse momentum); valid in lane 0
template <int LIM>
__device__ __forceinline__ void swe_edge_terms(const Row& row, int lane, const StepArgs& A, double ln, double lt,
                                               double am[3], double ap[3], double f[3])
{
    const double hg = 0.5 * A.grav;
    double h[4], n[4], t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        h[k] = row.at(0, k);
        n[k] = row.at(row.nm, k);
        t[k] = row.at(row.tm, k);
    }
    auto solve = [&](int k) { return swe_solve(h[k], n[k], t[k], h[k + 1], n[k + 1], t[k + 1], hg); };
    const bool second = A.order == 2;
    const double hw = (A.transverse == 2 && second) ? 1.0 : -1.0;
    const SEdge E = solve(1);
    double hp[3] = {0.0, 0.0, 0.0};
    if (second) swe_limited<LIM>(E, solve(0), solve(2), lane == 0 ? ln : lt, hp);
    const double s[3] = {E.un - E.c, E.un, E.un + E.c};
    const double a[3] = {E.a1, E.a2, E.a3};
    double cm[3] = {0.0, 0.0, 0.0}, cp[3] = {0.0, 0.0, 0.0};   // coefficients on r_p
    for (int p = 0; p < 3; ++p) {
        if (s[p] < 0.0) cm[p] = s[p] * a[p];
        else cp[p] = s[p] * a[p];
    }
    auto vec = [&](const double c3[3], double out[3]) {   // sum_p c_p r_p, r = (1, un -/+ c, ut), (0, 0, 1)
        out[0] = c3[0] + c3[2];
        out[1] = fma(s[0], c3[0], s[2] * c3[2]);
        out[2] = fma(E.ut, c3[0] + c3[2], c3[1]);
    };
    vec(cm, am);
    vec(cp, ap);
    f[0] = f[1] = f[2] = 0.0;
    if (second) vec(hp, f);
    if (A.transverse) {
        // the transverse sweep's fluctuations entering the cells either side, split along the normal: the
        // part of cell e-1 going to higher normal indices and the part of cell e going to lower ones
        // cross the edge
        double bm[3] = {0.0, 0.0, 0.0}, bp[3] = {0.0, 0.0, 0.0};
        swe_side_split(E, hp, lane == 1 || lane == 3, hw, bm, bp);
        double x[3];   // the transverse sweep's (h, its normal = our t, its tangential = our n)
#pragma unroll
        for (int m = 0; m < 3; ++m)
            x[m] = (lane_of(bp[m], 1) + lane_of(bp[m], 2)) + (lane_of(bm[m], 3) + lane_of(bm[m], 4));
        f[0] -= 0.5 * lt * x[0];
        f[1] -= 0.5 * lt * x[2];
        f[2] -= 0.5 * lt * x[1];
    }
}

// f(Q_F) - f(Q_C) of the shallow water equations along the edge's normal, (h, n, t) order
__device__ __forceinline__ void swe_flux_diff(const double qf[3], const double qc[3], int mn, double grav, double o[3])
{
    const int mt = 3 - mn;
    auto flux = [&](const double* v, double* fl) {
        const double ih = 1.0 / v[0];
        fl[0] = v[mn];
        fl[1] = fma(v[mn] * v[mn], ih, 0.5 * grav * v[0] * v[0]);
        fl[2] = v[mn] * v[mt] * ih;
    };
    double a[3], b[3];
    flux(qf, a);
    flux(qc, b);
    for (int m = 0; m < 3; ++m) o[m] = a[m] - b[m];
}

// edge-local (p, normal, transverse) -> (p, u, v)
__device__ __forceinline__ void to_puv(int dir, const double in[3], double out[3])
{
    out[0] = in[0];
    out[1] = dir == 0 ? in[1] : in[2];
    out[2] = dir == 0 ? in[2] : in[1];
}

// One edge of a job by eight lanes (item: the record, or record and fine edge, in range; on: its results
// are stored; all lanes of a warp call together).  Coarse: buf := minus the coarse part of the record and zero fine parts.
// Fine: slot (record, edge) of the fine part accumulates over the substeps (buf holds the coarse parts
// first, 3 per record, then the fine slots, 3 per record and edge).
template <int LIM>
__device__ __forceinline__ void edge_item(const RefluxJob& J, const StepArgs& A, int item, bool on)
{
    const int lane = threadIdx.x & 7;
    const int r = J.fine ? item / J.ratio : item, b = J.fine ? item - r * J.ratio : 0;
    const RefluxRec R = J.recs[r];
    const PatchDev C = J.cp[R.cbox];
    const PatchDev P = J.fine ? J.fp[R.fbox] : C;   // the box of the edge
    const double* q = (J.fine ? J.qf : J.qc) + P.qoff;
    const int W = P.nx + 4;
    const long long WH = (long long)W * (P.ny + 4);
    const double d = __ldg(A.dt + P.run) * P.dtscale;
    const double lx = d * P.dxinv, ly = d * P.dyinv;
    const double ln = R.dir == 0 ? lx : ly, lt = R.dir == 0 ? ly : lx;
    const int mn = R.dir == 0 ? 1 : 2;
    int cn, cl;   // the cell the record names on this level: normal index and line
    if (J.fine) {
        const int fi = R.dir == 0 ? R.fi : R.fi + b, fj = R.dir == 0 ? R.fj + b : R.fj;
        cn = R.dir == 0 ? fi : fj;
        cl = R.dir == 0 ? fj : fi;
    } else {
        cn = R.dir == 0 ? R.ci : R.cj;
        cl = R.dir == 0 ? R.cj : R.ci;
    }
    // C's east / north edge or its west / south edge; the fine cell's edge towards C
    const int e = (R.side > 0) != (J.fine != 0) ? cn + 1 : cn;
    const Row row(q, W, WH, R.dir, e, cl, lane);
    double am[3], ap[3], f[3], t[3], o[3];
    if (A.swe) swe_edge_terms<LIM>(row, lane, A, ln, lt, am, ap, f);
    else edge_terms<LIM>(row, lane, A, ln, lt, am, ap, f);
    if (!J.fine) {
        for (int m = 0; m < 3; ++m) t[m] = (R.side > 0 ? am[m] : -ap[m]) + f[m];
        to_puv(R.dir, t, o);
        if (!on) return;
        if (lane == 0)
            for (int m = 0; m < 3; ++m) J.buf[3 * r + m] = -o[m];
        for (int k = lane; k < 3 * J.ratio; k += kLanes) J.buf[3 * (J.n + r * J.ratio) + k] = 0.0;
        return;
    }
    if (!on || lane != 0) return;
    const int Wc = C.nx + 4;
    const long long WHc = (long long)Wc * (C.ny + 4);
    const long long co = C.qoff + (long long)(R.cj + 2) * Wc + (R.ci + 2);
    double qC[3], fl3[3];
    for (int m = 0; m < 3; ++m) qC[m] = J.qc[co + m * WHc];
    const int fi = R.dir == 0 ? cn : cl, fj = R.dir == 0 ? cl : cn;
    const double* qF_ = q + (long long)(fj + 2) * W + (fi + 2);
    if (A.swe) {
        const double qF[3] = {qF_[0], qF_[WH], qF_[2 * WH]};
        swe_flux_diff(qF, qC, mn, A.grav, fl3);   // f(Q_F) - f(Q_C) in the edge's order
    } else {
        // A (Q_F - Q_C) in the edge's order: (K dn, dp / rho, 0)
        const double dp = qF_[0] - qC[0], dn = qF_[mn * WH] - qC[mn];
        fl3[0] = A.K0 * dn;
        fl3[1] = dp * A.irho;
        fl3[2] = 0.0;
    }
    for (int m = 0; m < 3; ++m) t[m] = fl3[m] + (R.side > 0 ? -ap[m] : am[m]) + f[m];
    to_puv(R.dir, t, o);
    double* slot = J.buf + 3 * (J.n + item);
    for (int m = 0; m < 3; ++m) slot[m] += o[m];
}

__host__ __device__ inline int job_items(const RefluxJob& J) { return J.fine ? J.n * J.ratio : J.n; }

// the reflux jobs of a launch, by its CTAs [first, first + ctas) of NT threads
template <int LIM, int NT> __device__ __noinline__ void run_jobs(const StepArgs& A, int first, int ctas)
{
    const int n0 = job_items(A.reflux[0]), n = n0 + (A.nreflux > 1 ? job_items(A.reflux[1]) : 0);
    constexpr int per = NT / kLanes;
    for (int base = ((int)blockIdx.x - first) * per; base < n; base += ctas * per) {
        // (a warp may hold edges of both jobs: lanes exchange within their eight only)
        const int item = base + (int)threadIdx.x / kLanes;
        const bool on = item < n;
        // (lanes past the last edge run along on the first edge of a job that has one)
        const bool second = on ? item >= n0 : n0 == 0;
        edge_item<LIM>(A.reflux[second ? 1 : 0], A, on ? (second ? item - n0 : item) : 0, on);
    }
}

}  // namespace refl
}  // namespace claw
