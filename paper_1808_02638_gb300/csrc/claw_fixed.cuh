// claw_fixed.cuh -- one tile of the uniform-medium level-step in 64-bit fixed point.
//
// Why: this part issues about 1.7 FP64 instructions per SM and clock but 64 integer ones on its ALU
// pipe (measured: DADD 1.81, IADD3 121, LOP3 65, IMAD.WIDE 16 per SM and clock), so a double
// costs as much as some 35 integer instructions.  Between the jumps of q and the update of q the
// uniform-medium step is sums, comparisons and products with a few constants of the tile: with
// the tile's values scaled by one power of two they are 64-bit integers, a sum is two instructions
// and a product with a constant three wide multiplications.  FP64 is left where it is exact or
// where the result is formed: the jumps dp, du, dv (rounded as before) and q + increment (one
// fused multiply-add per component).
//
// Precision: with e such that |du|, |dv|, |dp| / Z < 2^e on every edge of the tile, by their exponents and that
// of 1 / Z, the unit is 2^(e - 58).  Sums and limiters are exact (van Leer's quotient within 7 units of
// M, see below), a product errs by at most one unit.  An increment of p / Z, u or v errs by up to 5
// units, 1.3 rms (emulated, uniformly random states with exact jumps: all limiters, orders and
// transverse modes); adding up every bound gives some 40.
//
// A tile is stepped this way only if at every edge the state next to it or the jump across it, the largest
// of |p| / Z, |u| and |v|, is at least 2^(e - 4): 5 units are then 2.5 roundings (2^-53) of that state, and
// the fused multiply-add that forms the result is the one other.  The FP64 phases take five such
// operations for p and three for u and v.  Emulated, relative to the state, in cells beside a
// jump at that limit: at most 2.5 and 1.7 roundings (p; u and v), 0.72 and 0.59 rms, where the FP64 phases
// have 4.4 and 2.9, 1.2 and 0.94.  The first-order step has two and one operations without transverse
// terms (2.0 and 1.0 roundings at most; fixed point 1.8 and 1.2 at 2^(e - 4)): it takes fixed point
// from 2^(e - 2) on.
//
// The precision is that of the state as a vector in wave units.  A component far smaller than the others and
// than the tile's jumps (a transverse velocity of 1e-9 beside jumps of 0.1 in p) is stepped to the same
// absolute error, 2^-56 of the largest jump, not to its own last bits as in FP64.
//
// Every other tile (a front on a zero background, infinities, NaN, extreme exponents, a CFL number above 1 in
// either direction) takes the FP64 phases, 2.6 times as long; a tile without any jump does not, whatever its
// state.  Path and unit depend on the states of the tile alone: how it was staged or who stepped it does
// not matter, but its shape does.  Two tilings of the same state agree to rounding, not bit for bit.
//
// What bounds it: the latency of dependent integer chains at 16 warps an SM; no pipe is at its limit (the ALU
// is the busiest), and FP64 and memory no longer are.  2048^2 in patches of 32^2 with pulled ghosts, MC
// limiter: 412 us a step when all of it was FP64, 185 now; 1001 x 604 in ragged patches, van Leer: 146 and
// 47 (the FP64 reciprocals went).
#pragma once

#include "claw_internal.h"

namespace claw {
namespace fx {

// ------------------------------------------------------------------------- numbers
// a constant c in [0, 1/4]: c = (hi 2^32 + lo) / 2^64, hi <= 2^30
struct __align__(16) Coef {
    unsigned hi, lo;
    unsigned half;   // 2^31 + lo / 2: half a unit, and the mean of the product that mul drops
};
__device__ __forceinline__ Coef coef_bits(long long c)   // c 2^64, at most 2^62
{
    Coef r;
    r.lo = (unsigned)c;
    r.hi = (unsigned)(c >> 32);
    r.half = 0x80000000u + (r.lo >> 1);
    return r;
}

// Rounding: products and conversions are of magnitudes, to nearest, and take the sign afterwards; quarters
// round halves to even.  Results are then odd functions of their arguments, so that a mirror-symmetric
// state stays so bit for bit, and their errors have no preferred sign.  Rounding downwards instead let
// the total of p drift by 6e-15 a step on 64^2 cells, linearly; like this it wanders no further than that
// of the FP64 phases.  (2048^2 took the same time so, 1001 x 604 with van Leer 44 us against 47.)

// w c for a magnitude w < 2^63, within a unit: the product of the low words, below one, is replaced by its mean.
// 0 gives 0: where nothing changes, nothing may.  (All unsigned: with a signed lo, whose sum of cross products
// is signed too, 2048^2 took 192 us a step, 185 so.)
__device__ __forceinline__ long long mul_mag(long long w, Coef c)
{
    const unsigned wh = (unsigned)(w >> 32);
    unsigned long long x = (unsigned long long)wh * c.lo + c.half;   // cross products, units / 2^32: below 2^63 + 2^62
    x += (unsigned long long)(unsigned)w * c.hi;
    return (long long)((unsigned long long)wh * c.hi + (x >> 32));
}
// m with its sign changed if s < 0.  (A select: exclusive or and difference took 203 against 194 us a step of
// 2048^2.)
__device__ __forceinline__ long long signed_by(long long m, int s) { return s < 0 ? -m : m; }
__device__ __forceinline__ int sign_of(long long v) { return (int)(v >> 32); }
__device__ __forceinline__ int sign_of(double d) { return __double2hiint(d); }
__device__ __forceinline__ long long mul(long long v, Coef c)
{
    const int s = sign_of(v);
    return signed_by(mul_mag(signed_by(v, s), c), s);
}
// v / 4, halves to even
__device__ __forceinline__ long long quarter(long long v) { return (v + 1 + ((v >> 2) & 1)) >> 2; }

__device__ __forceinline__ unsigned mag_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// |d| 2^(L + 1075 - base) for a finite d whose biased exponent is at most base (base >= 64: zeros and
// subnormals give 0), to nearest (halves up) or truncated
template <int L, bool NEAREST> __device__ __forceinline__ long long mag_from_double(double d, int base)
{
    const int hi = __double2hiint(d);
    const int e = (hi >> 20) & 0x7ff;
    unsigned long long m =
        ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(d);
    m <<= NEAREST ? L + 1 : L;
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(base - e));   // clamps at 64: no test of the amount
    return (long long)(NEAREST ? (m + 1) >> 1 : m);
}

// the double nearest to v, |v| < 2^62 (halves away from zero)
__device__ __forceinline__ double to_double(long long v)
{
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int lz = __clzll((long long)a);   // 2 .. 64
    const unsigned long long m = ((a << ((lz - 1) & 63)) + 0x200ull) >> 10;   // in [2^52, 2^53]
    unsigned hi = (unsigned)(m >> 32) + ((unsigned)(1085 - lz) << 20);
    hi = a ? hi : 0u;
    hi |= (unsigned)(v >> 32) & 0x80000000u;
    return __hiloint2double((int)hi, (int)(unsigned)m);
}

// ------------------------------------------------------------------------- limiters
// Lim2<L>::f(x, y) = 2 phi(y / x) x for x >= 0 and y of either sign, exact (van Leer's quotient is rounded,
// see below): the limited strength of a = x with its neighbour upwind b = y, both with a's sign taken out.
template <int L> struct Lim2;
template <> struct Lim2<CLAW_LIM_NONE> {
    static __device__ __forceinline__ long long f(long long x, long long) { return x + x; }
};
template <> struct Lim2<CLAW_LIM_MINMOD> {
    static __device__ __forceinline__ long long f(long long x, long long y)
    {
        const long long r = (x < y ? x : y) << 1;
        return y < 0 ? 0 : r;
    }
};
template <> struct Lim2<CLAW_LIM_SUPERBEE> {
    static __device__ __forceinline__ long long f(long long x, long long y)
    {   // 2 max(min(x, 2 y), min(2 x, y))
        const long long x2 = x << 1, y2 = y << 1;
        const long long m1 = x < y2 ? x : y2, m2 = x2 < y ? x2 : y;
        const long long r = (m1 > m2 ? m1 : m2) << 1;
        return y < 0 ? 0 : r;
    }
};
template <> struct Lim2<CLAW_LIM_MC> {
    static __device__ __forceinline__ long long f(long long x, long long y)
    {   // min(x + y, 4 min(x, y))
        const long long t = x + y, q = (x < y ? x : y) << 2;
        const long long r = t < q ? t : q;
        return y < 0 ? 0 : r;
    }
};

// 4 x y / (x + y) for x, y > 0: with s = x + y shifted to [2^60, 2^61), a reciprocal of its upper 32 bits
// (a float's 23 bits from below and one Newton step), the fraction f = min(x, y) / s in two digits of
// that reciprocal with the exact remainder between them, and 4 max(x, y) f.  f errs by less than
// 2^-60, the result (at most 2^60) by at most seven units; an integer or FP64 division would cost
// several times the 65 instructions.
template <> struct Lim2<CLAW_LIM_VANLEER> {
    static __device__ __forceinline__ long long f(long long x, long long y)
    {
        const unsigned long long lo = (unsigned long long)(x < y ? x : y), hi = (unsigned long long)(x < y ? y : x);
        const int sh = __clzll((long long)(lo + hi)) - 3;   // x + y < 2^60 and not 0 where the result is used
        const unsigned long long sn = (lo + hi) << (sh & 63), ln = lo << (sh & 63);
        const unsigned d = (unsigned)(sn >> 29);   // [2^31, 2^32)
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"((float)d));
        const unsigned v0 = (unsigned)(r * 9.2233676e18f);   // 2^63 / d less about 2^-20.9 of it
        const unsigned long long e = (1ull << 63) - (unsigned long long)v0 * d;
        const unsigned v = v0 + (__umulhi((unsigned)(e >> 11), v0) >> 20);
        const unsigned q1 = __umulhi((unsigned)(ln >> 29), v);   // f 2^31
        const unsigned long long p1 =
            (unsigned long long)q1 * (unsigned)sn + ((unsigned long long)(q1 * (unsigned)(sn >> 32)) << 32);
        const long long rem = (long long)((ln << 31) - p1);      // (f 2^31 - q1) sn, |.| < 2^63
        const long long p2 = (long long)(int)(rem >> 32) * (int)(v >> 1);   // rem / sn 2^59
        const unsigned long long f = ((unsigned long long)q1 << 31) + (unsigned long long)(p2 >> 28);   // f 2^62
        const unsigned long long h = hi << 4;
        const unsigned hh = (unsigned)(h >> 32), hl = (unsigned)h, fh = (unsigned)(f >> 32), fl = (unsigned)f;
        const unsigned c = __umulhi(hh, fl) + __umulhi(hl, fh);   // below 2^31 each
        const long long m = (long long)((unsigned long long)hh * fh + c);   // 4 max(x, y) f
        return x > 0 && y > 0 ? m : 0;
    }
};

// c 2 phi(b / a) a
template <int L> __device__ __forceinline__ long long limited(long long a, long long b, Coef c)
{
    const int s = sign_of(a);
    return signed_by(mul_mag(Lim2<L>::f(signed_by(a, s), signed_by(b, s)), c), s);
}

// ------------------------------------------------------------------------- shared state of a CTA
struct Shared {
    unsigned mp[2], mu[2];   // per tile parity: largest high words of |dp|, of |du| and |dv|
    int mn[2];               // smallest high word of the local magnitude of an edge (wave units)
    int iz_exp;              // 1 / Z0 = f 2^iz_exp, f in [1, 2); iz = f / 32
    Coef iz;
    // constants of a run, written by the last warp; two sets, so that one can be written while the
    // CTA's other threads finish a tile with the other
    struct Run {
        Coef c[6];           // see C_DX ..; nu = dt c0 / h
        double nux, nuy;
        int steep;           // 0: nu_x = nu_y, 1: nu_x larger, 2: nu_y larger
        int ok;              // 0 <= nu <= 1 in both directions, 1 / Z0 of a moderate exponent
    } run[2];
};
// (1 - nu_x) / 4, (1 - nu_y) / 4, nu_x / 4, nu_y / 4, the smaller of the two nu over four, the quotient of
// the smaller by the larger over four
enum : int { C_DX = 0, C_DY, C_NX, C_NY, C_MIN, C_RATIO };

__device__ __forceinline__ void init(Shared& S, double iZ)
{
    S.mp[0] = S.mp[1] = S.mu[0] = S.mu[1] = 0u;
    S.mn[0] = S.mn[1] = 0x7fffffff;
    const long long b = __double_as_longlong(iZ);
    S.iz_exp = (int)((b >> 52) & 0x7ff) - 1023;
    S.iz = coef_bits(((b & 0xfffffffffffffLL) | (1LL << 52)) << 7);
}

// by a whole warp, a lane per constant (one thread forming all of them held up a lone tile by 3800
// cycles, most of a third of it)
__device__ __forceinline__ void init_run(const Shared& S, Shared::Run& R, double dt, double dxinv, double dyinv,
                                         double c0)
{
    const int lane = threadIdx.x & 31;
    const double nu = dt * (lane & 1 ? dyinv : dxinv) * c0;
    const double nux = __shfl_sync(0xffffffffu, nu, 0), nuy = __shfl_sync(0xffffffffu, nu, 1);
    const bool in = nux >= 0.0 && nux <= 1.0 && nuy >= 0.0 && nuy <= 1.0;
    const double hi = nux > nuy ? nux : nuy, lo = nux > nuy ? nuy : nux;
    double v = lane < C_NX ? 1.0 - nu : lane < C_MIN ? nu : lo;
    if (hi != lo) v = lane == C_RATIO ? lo / hi : v;
    if (lane < 6 && in) R.c[lane] = coef_bits((long long)(v * 4611686018427387904.0));   // v / 4 2^64
    if (lane == 0) {
        R.ok = in && S.iz_exp > -400 && S.iz_exp < 400;
        R.nux = nux;
        R.nuy = nuy;
        R.steep = nux == nuy ? 0 : nux > nuy ? 1 : 2;
    }
}

// ------------------------------------------------------------------------- the tile
// Layout: the tile's positions are the cells a in [-1, tx + 1], r in [-1, ty + 1], each with its west
// x-edge and its south y-edge.  A thread takes one column a and a strip of up to R consecutive rows,
// and keeps everything of its positions in registers (no index arithmetic per edge); what a
// neighbour needs is exchanged through shared memory in slots [row of the strip][thread], where the
// column beside is the next thread and the strip above is w = tx + 3 threads further.
template <int TX, int TY, int NT> struct Strips {
    static constexpr int W = TX + 3, H = TY + 3;
    static constexpr int R = (H + NT / W - 1) / (NT / W);   // rows a thread takes at most
    // exchange slots in 8-byte words: strengths a1, a2 (later E and the ends' D), limited S, P
    // (R rows each), and of each strip b1 and b2 at its ends, limited y-edge S and P at its bottom
    static constexpr int WORDS = (4 * R + 4) * NT + 2;
};

// the value of the row above / below row j of a strip of `rows` rows; `next` / `prev`: the strip beside
template <int R> __device__ __forceinline__ long long above(const long long (&x)[R], int j, int rows, long long next)
{
    if (j + 1 >= R) return next;
    const long long y = x[j + 1 < R ? j + 1 : 0];
    return j + 1 < rows ? y : next;
}
template <int R> __device__ __forceinline__ long long below(const long long (&x)[R], int j, long long prev)
{
    if (j == 0) return prev;
    return x[j > 0 ? j - 1 : 0];
}

// row rows - 1 of a strip, by selects (a register array is not indexed)
template <int R> __device__ __forceinline__ long long last_row(const long long (&x)[R], int rows)
{
    long long y = x[0];
#pragma unroll
    for (int j = 1; j < R; ++j)
        if (j < rows) y = x[j];
    return y;
}

// Steps the staged tile (planes sp, su, sv = sq, sq + QPL, sq + 2 QPL) into q_new and returns true,
// or returns false with nothing written and the tile still staged (uniform over the CTA).  KEEP: the
// staged tile is read before the first barrier only (the next tile's copy may land in it behind
// that); otherwise it is read again at the end.  `jumps_done` is called before the
// first barrier and, on the fixed-point path, `begin` behind it, `strengths_done` before the
// second and `limited_done` before the third: the fetches for the next tile.  What the last phase reads of
// the exchange slots is next written behind two barriers of the next tile, so no barrier ends the tile.
//
// Units and ranges, U = 2^58 the bound of |du|, |dv|, |dp| / Z and A = 2 U that of the strengths:
//   a1, a2 = du -+ dp / Z                                          A = 2^59
//   M = (1 - nu) / 4 2 phi a, S = M2 - M1, P = M1 + M2             A
//   ap = A2_w + A1_e, au = A2_w - A1_e                             2 A
//   m = S_e - S_w, n = P_e - P_w   (k, l of the y-edges)           2 A
//   D / 4 = (ap + 2 m) / 4  (x-fluctuation pressure; E likewise)   3/2 A
//   X = ap + m, U = au + n of the x-edges, Y, V of the y-edges    4 A
// and with Q4 = (D_n + D_s - 2 D + E_e + E_w - 2 E) / 4 (below 12 A < 2^63) the increments are
//   p / Z  -1/2 (nu_x X + nu_y Y + nu_x nu_y Q4)
//   u      -nu_x / 2 (U - nu_y (E_e - E_w) / 4),   v  -nu_y / 2 (V - nu_x (D_n - D_s) / 4)
// The larger nu of p and the nu in front of u and v are left to the fused multiply-add that adds the
// increment to q (in FP64, with the bracket, of p a quarter of it, as its integer operand: below 5 A
// and 7 A), so that square cells take no product for them and others one.  4 (E_e - E_w) is below 12 A.
template <class G, int LIM, int TX, int TY, int NT, bool KEEP, class Jumps, class Begin, class Strengths,
          class Limited>
__device__ __forceinline__ bool step_tile(const StepArgs& A, const PatchDev& P, Shared& sh, const Shared::Run& run,
                                          int par, const double* sp, double* work, double Z0, int tx, int ty, int x0,
                                          int y0, int& my_flag, Jumps jumps_done, Begin begin,
                                          Strengths strengths_done, Limited limited_done)
{
    using T = Strips<TX, TY, NT>;
    constexpr int R = T::R;
    long long* A1 = reinterpret_cast<long long*>(work) + 1 + threadIdx.x;   // this thread's slots
    long long* A2 = A1 + R * NT;
    long long* SX = A2 + R * NT;
    long long* PX = SX + R * NT;
    long long* B1 = PX + R * NT;   // b1 of the strip's first row
    long long* B2 = B1 + NT;       // b2 of its last
    long long* SY = B2 + NT;       // limited y-edge of its first row
    long long* PY = SY + NT;
    const int tid = threadIdx.x;
    const bool second = A.order == 2;
    const bool trans = A.transverse != 0;
    const bool cw = A.transverse == 2 && A.order == 2;
    // (rows past a strip's last compute on zeros in slots of their own; only their global stores are left out)

    const int w = tx + 3, h = ty + 3;
    const int strips = NT / w;                       // strips side by side in the CTA
    const int rows = (h + strips - 1) / strips;      // rows of a strip, at most R
    const int strip = tid / w, a = tid - strip * w - 1, r0 = strip * rows - 1;
    // rows of this thread (strips past the tile's last row and the last threads take none)
    const int nr = strip < strips ? min(rows, h - 1 - r0) : 0;
    const bool up = r0 + rows <= ty + 1;             // another strip continues this one

    // ---------------------------------------------------------------- jumps (FP64) and their scale
    double xp[R], xu[R], yp[R], yv[R], q[KEEP ? R : 1][3];
    {
        unsigned mp = 0u, mu = 0u;
        int mn = 0x7fffffff;
        const int izs = sh.iz_exp << 20;
        const double* s = sp + (a + 2) + (r0 + 2) * G::SW;
        double ps = 0.0, vs = 0.0;   // the cell below
        if (nr > 0) {
            ps = s[-G::SW];
            vs = s[2 * G::QPL - G::SW];
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const bool in = j < nr, ex = in && r0 + j <= ty, ey = in && a <= tx;
            double p = 0.0, u = 0.0, v = 0.0, pw = 0.0, uw = 0.0;
            if (in) {
                p = s[j * G::SW];
                u = s[G::QPL + j * G::SW];
                v = s[2 * G::QPL + j * G::SW];
                pw = s[j * G::SW - 1];
                uw = s[G::QPL + j * G::SW - 1];
            }
            xp[j] = p - pw;
            xu[j] = u - uw;
            yp[j] = p - ps;
            yv[j] = v - vs;
            const unsigned jp = max(ex ? mag_hi(xp[j]) : 0u, ey ? mag_hi(yp[j]) : 0u);
            const unsigned ju = max(ex ? mag_hi(xu[j]) : 0u, ey ? mag_hi(yv[j]) : 0u);
            mp = max(mp, jp);
            mu = max(mu, ju);
            // the state's and the jumps' magnitude at this position in wave units (an exponent
            // field that overflows turns negative, which sends the tile to the FP64 phases)
            const int m = max((int)max(ju, max(mag_hi(u), mag_hi(v))), (int)max(jp, mag_hi(p)) + izs);
            mn = ex || ey ? min(mn, m) : mn;
            ps = p;
            vs = v;
            if (KEEP) {
                q[j][0] = p;
                q[j][1] = u;
                q[j][2] = v;
            }
        }
        mp = __reduce_max_sync(0xffffffffu, mp);
        mu = __reduce_max_sync(0xffffffffu, mu);
        mn = __reduce_min_sync(0xffffffffu, mn);
        if ((tid & 31) == 0) {
            atomicMax(&sh.mp[par], mp);
            atomicMax(&sh.mu[par], mu);
            atomicMin(&sh.mn[par], mn);
        }
    }
    jumps_done();
    __syncthreads();
    const unsigned mp = sh.mp[par], mu = sh.mu[par];
    const int mn = sh.mn[par];
    if (tid == 0) {   // the next tile's slot; its last readers are behind this barrier
        sh.mp[par ^ 1] = sh.mu[par ^ 1] = 0u;
        sh.mn[par ^ 1] = 0x7fffffff;
    }
    // e: |du|, |dv|, |dp| / Z < 2^(e - 1022)
    int e = max((int)(mu >> 20), mp ? (int)(mp >> 20) + sh.iz_exp + 1 : 0);
    bool fine = run.ok && mp < 0x7ff00000u && mu < 0x7ff00000u;
    if ((mp | mu) == 0u) e = 1023;   // no jump above 2^-1042: every fixed-point jump is 0
    const int least = second ? e - 3 : e - 1;   // biased exponent: 2^(e - 4) and 2^(e - 2) of the bound
    fine = fine && e >= 500 && e <= 1600 && (mn >> 20) >= ((mp | mu) ? least : 100);
    if (!fine && run.ok && (mp | mu) == 0u) {
        // a tile whose jumps are zero to the last bit comes out as it is, in integers as in FP64, however small its
        // state.  (Zeros in front of a wave, the whole of 2048^2: 507 us by the FP64 phases, 211 so.)
        bool still = true;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const bool in = j < nr;
            if (in && r0 + j <= ty) still = still && xp[j] == 0.0 && xu[j] == 0.0;
            if (in && a <= tx) still = still && yp[j] == 0.0 && yv[j] == 0.0;
        }
        fine = !__syncthreads_or(!still);
    }
    if (!fine) return false;
    begin();

    // ---------------------------------------------------------------- strengths a1, a2 = du -+ dp / Z
    long long a1[R], a2[R], b1[R], b2[R];
    {
        const int bp = e - sh.iz_exp - 1;   // biased exponent bound of dp
        const Coef iz = sh.iz;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const long long tx_ = signed_by(mul_mag(mag_from_double<9, false>(xp[j], bp), iz), sign_of(xp[j]));
            const long long dx = signed_by(mag_from_double<5, true>(xu[j], e), sign_of(xu[j]));
            a1[j] = dx - tx_;
            a2[j] = dx + tx_;
            A1[j * NT] = a1[j];
            A2[j * NT] = a2[j];
            const long long ty_ = signed_by(mul_mag(mag_from_double<9, false>(yp[j], bp), iz), sign_of(yp[j]));
            const long long dy = signed_by(mag_from_double<5, true>(yv[j], e), sign_of(yv[j]));
            b1[j] = dy - ty_;
            b2[j] = dy + ty_;
        }
        B1[0] = b1[0];
        B2[0] = last_row(b2, rows);
    }
    strengths_done();
    __syncthreads();

    // ---------------------------------------------------------------- limited strengths
    long long ap[R], au[R], bp[R], bv[R], sy[R] = {}, py[R] = {};
    {
        const long long b1u = up ? B1[w] : 0, b2d = strip > 0 ? B2[-w] : 0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const long long a1e = A1[j * NT + 1];
            const long long b1n = above(b1, j, rows, b1u);
            ap[j] = a2[j] + a1e;
            au[j] = a2[j] - a1e;
            bp[j] = b2[j] + b1n;
            bv[j] = b2[j] - b1n;
            if (second) {
                const Coef cx = run.c[C_DX], cy = run.c[C_DY];
                const long long m1 = limited<LIM>(a1[j], a1e, cx);   // left-going: upwind edge to the right
                const long long m2 = limited<LIM>(a2[j], A2[j * NT - 1], cx);
                SX[j * NT] = m2 - m1;
                PX[j * NT] = m1 + m2;
                const long long n1 = limited<LIM>(b1[j], b1n, cy);
                const long long n2 = limited<LIM>(b2[j], below(b2, j, b2d), cy);
                sy[j] = n2 - n1;
                py[j] = n1 + n2;
                if (j == 0) {
                    SY[0] = sy[0];
                    PY[0] = py[0];
                }
            }
        }
    }
    limited_done();
    __syncthreads();

    // ---------------------------------------------------------------- per-cell terms
    // the exchange slots of a1, a2 are free: E goes to A1, D of a strip's first and last row to A2
    long long hp[R], hu[R], hv[R], d4[R], e4[R];   // the brackets (of p: a quarter); D / 4, E / 4
    {
        const long long syu = second && up ? SY[w] : 0, pyu = second && up ? PY[w] : 0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            long long m = 0, n = 0, k = 0, l = 0;
            if (second) {
                m = SX[j * NT + 1] - SX[j * NT];
                n = PX[j * NT + 1] - PX[j * NT];
                k = above(sy, j, rows, syu) - sy[j];
                l = above(py, j, rows, pyu) - py[j];
            }
            const long long X = ap[j] + m, Y = bp[j] + k;
            if (run.steep == 0) hp[j] = quarter(X + Y);
            else if (run.steep == 1) hp[j] = quarter(X) + mul(Y, run.c[C_RATIO]);
            else hp[j] = quarter(Y) + mul(X, run.c[C_RATIO]);
            hu[j] = au[j] + n;
            hv[j] = bv[j] + l;
            d4[j] = quarter(ap[j] + (cw ? m + m : 0));
            e4[j] = quarter(bp[j] + (cw ? k + k : 0));
            if (trans) {
                A1[j * NT] = e4[j];
            }
        }
        if (trans) {
            A2[0] = d4[0];
            A2[NT] = last_row(d4, rows);
        }
    }
    if (trans) __syncthreads();

    // ---------------------------------------------------------------- update, store
    if (nr > 0 && a >= 0 && a < tx) {
        const double unit2 = -__hiloint2double((e - 56) << 20, 0);   // -2^(e - 1079), twice the unit
        const double kx = run.nux * unit2, ky = run.nuy * unit2;
        const double kp = Z0 * (run.steep == 2 ? ky : kx), ku = 0.25 * kx, kv = 0.25 * ky;
        const int W = P.nx + 4;
        const long long WH = (long long)W * (P.ny + 4);
        double* dst = A.qnew + P.qoff + (long long)(y0 + r0 + 2) * W + (x0 + a + 2);
        const long long du = trans && up ? A2[w] : 0, dd = trans && strip > 0 ? A2[NT - w] : 0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            if (j >= nr || r0 + j < 0 || r0 + j >= ty) continue;
            if (trans) {
                const long long dn = above(d4, j, rows, du);
                const long long ds = below(d4, j, dd);
                const long long ee = A1[j * NT + 1], ew = A1[j * NT - 1];
                hp[j] += mul((dn + ds) + (ee + ew) - 2 * (d4[j] + e4[j]), run.c[C_MIN]);
                hu[j] -= mul((ee - ew) << 2, run.c[C_NY]);
                hv[j] -= mul((dn - ds) << 2, run.c[C_NX]);
            }
            const double* s = sp + (a + 2) + (r0 + j + 2) * G::SW;
            const double p = fma(to_double(hp[j]), kp, KEEP ? q[KEEP ? j : 0][0] : s[0]);
            const double u = fma(to_double(hu[j]), ku, KEEP ? q[KEEP ? j : 0][1] : s[G::QPL]);
            const double v = fma(to_double(hv[j]), kv, KEEP ? q[KEEP ? j : 0][2] : s[2 * G::QPL]);
            if (max(mag_hi(p), max(mag_hi(u), mag_hi(v))) >= 0x7ff00000u) my_flag |= ERR_NAN;
            dst[(long long)j * W] = p;
            dst[(long long)j * W + WH] = u;
            dst[(long long)j * W + 2 * WH] = v;
        }
    }
    return true;
}

}  // namespace fx
}  // namespace claw
