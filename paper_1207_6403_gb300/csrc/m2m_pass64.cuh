// The FP64 particle pass.
//
// An FP64 warp instruction takes 16 cycles of an SM here (an FP32 one a
// quarter of a cycle), so the pass is bound by the number of double
// operations per particle, not by memory (120 of 200 to 240 bytes moved are the
// step's own and take a twentieth of the time).  What follows from that:
//  - inside one m2m_step call a pass leaves what the next one would compute
//    again from the same particle: the force at the new position, ln(w/w_hat)
//    of the stored weight (see log_carry) and, per Gauss-Hermite set, m and
//    the Gaussian factor of the cell the scatter found (56 bytes per particle,
//    PassArgs c64); m2m_step alone sets the flags, so a caller may change its
//    arrays between calls as before;
//  - cells are decided on the doubles' bit patterns (order-preserving integer
//    keys, exactly the double comparisons) and the float index guess comes
//    from the bits, so a bin search has no FP64 instruction;
//  - an expansion's force is a call (m2m_device.cuh, ex_accel_call);
//  - exp is table driven (P. T. P. Tang, ACM TOMS 15 (1989) 144: exp(x) =
//    2^(k/128) exp(r), |r| <= ln 2/256, a quintic in r), 10 operations; the
//    weight's exp(d) is 1 + its series, to d^5 for |d| < 2^-10 and to d^8 for
//    |d| < 2^-5 (what is left out is below 2^-58 of d);
//  - the moments are polynomials of m with the constants of gh_record, no
//    division;
//  - a double shared-memory add is a compare-and-swap loop, which the lanes
//    of a warp that share a bin run one after the other: lanes add to copies
//    of their own where the bins leave room (hist_copies), and the block's
//    sums go into the double totals with global atomics;
//  - warps are dealt chunks of 32 particles round the blocks, so that a small
//    model occupies every SM.
// 300,000 particles, pixels + apertures in the logarithmic potential: a step
// takes 111 us, 454 before; 20,000 particles, shells + annuli, 22 us, 125
// before.  Global double atomics instead of the shared histogram were slower
// (300,000 particles 139 us a step, shells + annuli at 200,000 276 against 79:
// many particles share a total).
#pragma once
#include "m2m_kernels.cuh"

namespace m2m {

constexpr int EXP_N = 128;           // entries 2^(j/128) of the exp table

// Order-preserving integer key of a double that is not NaN; -0 as +0.
__device__ __forceinline__ long long dkey(double v) {
    const long long b = __double_as_longlong(v);
    return (b << 1) == 0 ? 0ll : b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// The float nearest a double towards zero, from its bits (infinite above the
// float range; integer instructions only, also for subnormal floats).
__device__ __forceinline__ float d2f_bits(double v) {
    const unsigned hi = (unsigned)__double2hiint(v);
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;                     // float biased exponent
    const unsigned m = __funnelshift_l((unsigned)__double2loint(v), hi, 3) & 0x7fffffu;
    unsigned r = e > 0 ? ((unsigned)e << 23) | m : __funnelshift_rc(m | 0x800000u, 0u, (unsigned)(1 - e));
    r = e >= 255 ? 0x7f800000u : r;
    return __uint_as_float(r | (hi & 0x80000000u));
}

// find_fast on keys: the guess is within a cell of the true one, the keys of
// the guessed cell's two edges decide.
template <int MODE>
__device__ __forceinline__ int find_fast64(double v, const longlong2 *e, int nb, float ga, float gb, float top) {
    const float fv = d2f_bits(v);
    const float t = MODE == G_LOG ? __log2f(fv) : fv;
    int g = rint_small(fminf(fmaxf(fmaf(ga, t, gb) - 0.5f, 0.0f), top));
    const longlong2 ed = e[g];
    const long long k = dkey(v);
    g += (k >= ed.y ? 1 : 0) - (k < ed.x ? 1 : 0);
    const bool fin = (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;     // NaN and infinities: no cell
    return fin && (unsigned)g < (unsigned)nb ? g : -1;
}

template <int G>
__device__ __forceinline__ int cell64(const SetDev &s, const longlong2 *ek, double x, double y, double z, double X,
                                      double Ys) {
    if constexpr (G == M2M_GEOM_SHELL) {
        return find_fast64<G_LOG>((x * x + y * y) + z * z, ek + s.ex_off, s.nx, s.gx_a, s.gx_b, s.gx_top);
    } else if constexpr (G == M2M_GEOM_ANNULUS) {
        return find_fast64<G_LOG>(X * X + Ys * Ys, ek + s.ex_off, s.nx, s.gx_a, s.gx_b, s.gx_top);
    } else {
        const int ix = find_fast64<G_LIN>(X, ek + s.ex_off, s.nx, s.gx_a, s.gx_b, s.gx_top);
        const int iy = find_fast64<G_LIN>(Ys, ek + s.ey_off, s.ny, s.gy_a, s.gy_b, s.gy_top);
        return (ix < 0 || iy < 0) ? -1 : iy * s.nx + ix;
    }
}

// e^x for x <= 0 (0 below -700, NaN for NaN); T[j] = 2^(j/128).
__device__ __forceinline__ double exp_neg(double x, const double *T) {
    const unsigned hx = (unsigned)__double2hiint(x);
    const double n = fma(x, 184.66496523378731, 6755399441055744.0);   // 128/ln 2, 1.5 * 2^52
    const int k = __double2loint(n);
    const double nf = n - 6755399441055744.0;
    // ln 2/128 as the nearest double and the rest
    double r = fma(nf, -0.6931471805599453094 / 128.0, x);
    r = fma(nf, -2.3190468138462996e-17 / 128.0, r);
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(q, r, 1.0 / 6.0);
    q = fma(q, r, 0.5);
    const double p = fma(q * r, r, r);
    const double t = __ldg(T + (k & (EXP_N - 1)));
    const double e = fma(t, p, t);
    const double v = __hiloint2double(__double2hiint(e) + ((k >> 7) << 20), __double2loint(e));
    return hx - 0xC085E000u <= 0xFFF00000u - 0xC085E000u ? 0.0 : v;     // -inf <= x <= -700
}

// gh_eval in double for the run-time set walk: g = (V, 1/S, c1, t2, norm).
__device__ __forceinline__ void gh_eval(double vlos, const double *g, double u[5], const double *T) {
    const double SQ2 = 1.4142135623730951, K3 = 1.1547005383792515, K4 = 0.81649658092772603;
    const double nu = (vlos - g[0]) * g[1], m = nu * g[2], m2 = m * m, d = fma(2.0, g[3], -1.0);
    const double e = g[4] * exp_neg((nu * m) * -0.5, T);
    u[0] = e;
    u[1] = e * (SQ2 * m);
    u[2] = e * fma(SQ2, m2, d * 0.70710678118654752);
    u[3] = e * (m * fma(K3, m2, d * 1.7320508075688772));
    u[4] = e * fma(m2, fma(K4, m2, d * 2.4494897427831779), (d * d) * 0.61237243569579447);
}

struct Smem64 {
    double *h;               // histogram: [observable][copies] as hist_at
    int hrep, hlane;
    const double *coef, *edges, *gh, *gpoly;
    const longlong2 *ekey;   // keys of (e[k], e[k+1])
    PassSmem<double> cells;  // prior grid and cell sums
};

__device__ __forceinline__ void hist64(const Smem64 &S, int i, double v) { atomicAdd(S.h + i, v); }

// Gauss-Hermite cell of the compiled layouts (S.gh, 5 doubles): V, c1/S,
// -1/(2S), norm, d = 2 t2 - 1; S.gpoly: the update's quartic in m.
struct GhPoint { double m, g; };
__device__ __forceinline__ GhPoint gh_point(const double *r, double vlos, const double *T) {
    const double dv = vlos - r[0], m = dv * r[1];
    return {m, r[3] * exp_neg((dv * m) * r[2], T)};
}

// A weight far enough from the ends of the double range for log_carry.
__device__ __forceinline__ bool mid_weight(double w) {
    return ((unsigned)__double2hiint(w) >> 20) - 123u <= 1800u;          // 2^-900 .. 2^900
}

// ln(wn/w_hat) of the stored weight wn = w + w e (rounded; e = e^d - 1) from
// ln(w/w_hat) = L + l: L + d less what the rounding of wn took, rem/wn, as a
// sum and its remainder l (T. J. Dekker, Numer. Math. 18 (1971) 224, the
// larger term first by exponent).  L + d alone would not do: its roundings
// and the weights' add up over the steps of a call, and a weight that no
// longer moves (|d| below half an ulp) would leave the sum moving on.  As it
// is, the error after 4000 steps is that of one fresh logarithm (rms 6e-17;
// L + d alone 5e-15 and more).  Seven FP64 operations, where the quotient and
// the logarithm take 40: where half of the warps took those (a series and so
// the carry only below |d| = 2^-10), 300,000 particles, pixels + apertures, 25
// steps took 3210 us against 2820.
__device__ __forceinline__ double log_carry(double L, double &l, double w, double wn, double d, double e) {
    const double rem = fma(w, e, w - wn);            // the difference is exact (|e| < 2^-4)
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(wn));               // 20 bits: rem is below an ulp
    const double c = d + fma(-rem, y, l);
    const bool first = ((unsigned)__double2hiint(L) & 0x7fffffffu) >= ((unsigned)__double2hiint(c) & 0x7fffffffu);
    const double p = first ? L : c, q = first ? c : L, s = p + q;
    l = q - (s - p);
    return s;
}

// One pass over the particles of block `bid` of `nblk`.  L: compiled layout
// (1: pixels + apertures, 2: shells + GH annuli, 3: shells + mass and v^2
// annuli), 0: the run-time set walk.
template <int NT, int L>
__device__ __forceinline__ void pass64_body(const PassArgs &a, const int bid, const int nblk) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[32];
    const int fl = a.flags, nobs = a.nobs;
    Smem64 S{};
    PassSmem<double> &C = S.cells;
    unsigned char *p = smem;
    if (fl & F_SCAT) {
        S.hrep = a.hrep;
        S.hlane = (int)threadIdx.x & (a.hrep - 1);
        S.h = (double *)p; p += 8 * (size_t)a.hrep * ((nobs + 1) & ~1);
    }
    // the compiled layouts read the few coefficients a particle needs (one per
    // mass or v^2 set; the GH ones are in gpoly) from L2: the space goes to
    // the histogram's copies
    S.coef = (const double *)a.coef;
    if (L == 0 && (fl & F_UPD)) { S.coef = (const double *)p; p += 8 * ((nobs + 3) & ~3); }
    if (L == 0) { S.edges = (const double *)p; p += 8 * ((a.edge_len + 3) & ~3); }
    else { S.ekey = (const longlong2 *)p; p += 16 * ((a.edge_len + 1) & ~1); }
    S.gh = (const double *)p; p += 8 * ((a.gh_len + 3) & ~3);
    if (L != 0 && (fl & F_UPD)) { S.gpoly = (const double *)p; p += 8 * ((a.gh_len + 3) & ~3); }
    const int sh_len = (a.sh_tab && (fl & (F_PUSH | F_MINMAX | F_CELLS))) ? a.sh_row * a.sh_K : 0;
    const double *sh = nullptr;
    if (sh_len) { sh = (const double *)p; p += 8 * ((sh_len + 3) & ~3); }
    if (fl & F_CELLS) {
        C.pe = (double *)p; p += 8 * ((a.nE + 4) & ~3);
        C.pl = (double *)p; p += 8 * ((a.nL + 4) & ~3);
        C.gp = (float *)p; p += 16;
        C.c_d = (double *)p; p += 8 * ((a.ncells + 1) & ~1);
        C.c_lo = (unsigned *)p; p += 4 * ((a.ncells + 3) & ~3);   // counts
    }
    // fixed tables and cleared sums, then what a preceding kernel may write
    if (fl & F_SCAT)
        for (int k = threadIdx.x; k < nobs * a.hrep; k += NT) S.h[k] = 0.0;
    const double *et = (const double *)a.edge_tab;
    if constexpr (L == 0) {
        stage<2>((double *)S.edges, et, a.edge_len, threadIdx.x, NT);
        stage<2>((double *)S.gh, (const double *)a.gh_tab, a.gh_len, threadIdx.x, NT);
    } else {
        for (int k = threadIdx.x; k < a.edge_len; k += NT)
            ((longlong2 *)S.ekey)[k] = make_longlong2(dkey(et[k]), k + 1 < a.edge_len ? dkey(et[k + 1]) : LLONG_MAX);
    }
    griddep_wait();
    if (L == 0 && (fl & F_UPD)) stage<4>((double *)S.coef, (const double *)a.coef, nobs, threadIdx.x, NT);
    if (sh_len) stage<4>((double *)sh, (const double *)a.sh_tab, sh_len, threadIdx.x, NT);
    if constexpr (L != 0) {
        for (int k = 0; k < a.nsets; ++k) {
            const SetDev &st = a.sets[k];
            if (st.quant != M2M_Q_GH) continue;
            for (int c = threadIdx.x; c < st.ncell; c += NT) {
                const double *g = (const double *)a.gh_tab + st.gh_off + 5 * c;   // V, 1/S, c1, t2, norm
                double *r = (double *)S.gh + st.gh_off + 5 * c;
                r[0] = g[0]; r[1] = g[2] * g[1]; r[2] = -0.5 * g[1]; r[3] = g[4]; r[4] = fma(2.0, g[3], -1.0);
                if (fl & F_UPD) {
                    // gh_quartic without the norm, in d: no divisions (every
                    // block builds every cell's, which took 5 us of a pass)
                    const double *cf = (const double *)a.coef + st.obs_off + 5 * c;
                    double *P = (double *)S.gpoly + st.gh_off + 5 * c;
                    const double d = r[4], c2 = __ldcg(cf + 2), c3 = __ldcg(cf + 3), c4 = __ldcg(cf + 4);
                    P[0] = fma(c4, (d * d) * 0.61237243569579447, fma(c2, d * 0.70710678118654752, __ldcg(cf)));
                    P[1] = fma(c3, d * 1.7320508075688772, __ldcg(cf + 1) * 1.4142135623730951);
                    P[2] = fma(c4, d * 2.4494897427831779, c2 * 1.4142135623730951);
                    P[3] = c3 * 1.1547005383792515;
                    P[4] = c4 * 0.81649658092772603;
                }
            }
        }
    }
    if (fl & F_CELLS) {
        for (int k = threadIdx.x; k < a.ncells; k += NT) { C.c_d[k] = 0.0; C.c_lo[k] = 0u; }
        prior_setup<double>(a, C.pe, C.pl, C.gp);
    }
    __syncthreads();

    const double sn = a.sin_i, cs = a.cos_i;
    const double *T = a.exp_tab;
    const unsigned n = (unsigned)a.n, stride = (unsigned)nblk * NT;
    double *px = (double *)a.x, *py = (double *)a.y, *pz = (double *)a.z;
    double *pvx = (double *)a.vx, *pvy = (double *)a.vy, *pvz = (double *)a.vz;
    double s_d = 0.0, w_d = 0.0, emin = INFINITY, emax = -INFINITY, lzm = 0.0;
    bool bad = false, ovf = false;
    for (unsigned i = ((threadIdx.x >> 5) * (unsigned)nblk + (unsigned)bid) * 32u + (threadIdx.x & 31); i < n;
         i += stride) {
        double x = px[i], y = py[i], z = pz[i], vx = pvx[i], vy = pvy[i], vz = pvz[i];
        const double w = a.w[i];
        double wn = w;
        if (fl & (F_UPD | F_STATS)) {
            if (d_pos(w)) {
                double Lw, Ll = 0.0;          // ln(w/w_hat) and, kept, what its rounding left out
                if (a.c64_read & C64_LNW) { Lw = a.c64_lnw[i]; Ll = a.c64_lnl[i]; }
                else Lw = log(w / a.what[i]);
                double wr = w, Lk = Lw;       // Lk: what the next pass finds
                if (fl & F_UPD) {
                    double dot = 0.0;
                    if constexpr (L == 0) {
                        const double X = x, Ys = z * sn - y * cs, vlos = vy * sn + vz * cs;
                        for (int k = 0; k < a.nsets; ++k) {
                            const SetDev &s = a.sets[k];
                            double Xk = X, Yk = Ys;
                            if (s.psf) seeing<double>(s, k, i, a.epoch, Xk, Yk);
                            const int c = set_cell<double>(s, S.edges, x, y, z, Xk, Yk);
                            if (c < 0) continue;
                            const double *cf = S.coef + s.obs_off + c * s.nmom;
                            if (s.quant == M2M_Q_MASS) {
                                dot = dot + cf[0];
                            } else if (s.quant == M2M_Q_VLOS2) {
                                dot = dot + (vlos * vlos) * cf[0];
                            } else {
                                double u[5];
                                gh_eval(vlos, S.gh + s.gh_off + 5 * c, u, T);
#pragma unroll
                                for (int m = 0; m < 5; ++m) dot = fma(u[m], cf[m], dot);
                            }
                        }
                    } else {
                        const unsigned cc = a.cache_read ? a.cell_cache[i] : 0u;
                        for_each_set<L>([&](auto K, auto G, auto Q) {
                            constexpr int k = decltype(K)::value, g = decltype(G)::value, q = decltype(Q)::value;
                            const SetDev &s = a.sets[k];
                            const int c = a.cache_read ? (int)((cc >> s.cshift) & (unsigned)s.cmask) - 1
                                                       : cell64<g>(s, S.ekey, x, y, z, x, z * sn - y * cs);
                            if (c < 0) return;
                            if constexpr (q == M2M_Q_MASS) {
                                dot = dot + __ldcg(S.coef + s.obs_off + c);
                            } else if constexpr (q == M2M_Q_VLOS2) {
                                const double vlos = vy * sn + vz * cs;
                                dot = dot + (vlos * vlos) * __ldcg(S.coef + s.obs_off + c);
                            } else {
                                GhPoint h;
                                if (a.c64_read & C64_GH) h = {a.c64_m[i], a.c64_g[i]};
                                else h = gh_point(S.gh + s.gh_off + 5 * c, vy * sn + vz * cs, T);
                                const double *P = S.gpoly + s.gh_off + 5 * c;
                                double q4 = fma(P[4], h.m, P[3]);
                                q4 = fma(q4, h.m, P[2]);
                                q4 = fma(q4, h.m, P[1]);
                                q4 = fma(q4, h.m, P[0]);
                                dot = fma(h.g, q4, dot);
                            }
                        });
                    }
                    const double G = a.mu * (-Lw - a.ent_c) - dot;
                    const double d = a.eps_dt * G;
                    const unsigned dx = (unsigned)__double2hiint(d) & 0x7fffffffu;
                    double e = 0.0;
                    if (dx < 0x3FA00000u) {                      // |d| < 2^-5
                        e = 1.0 / 120.0;
                        if (dx >= 0x3F500000u) {                 // |d| >= 2^-10
                            e = fma(d, 1.0 / 40320.0, 1.0 / 5040.0);
                            e = fma(d, e, 1.0 / 720.0);
                            e = fma(d, e, 1.0 / 120.0);
                        }
                        e = fma(d, e, 1.0 / 24.0);
                        e = fma(d, e, 1.0 / 6.0);
                        e = fma(d, e, 0.5);
                        e = fma(d, e, 1.0);
                        e = d * e;                               // e^d - 1
                        wn = fma(w, e, w);
                    } else {
                        wn = w * exp(d);
                    }
                    wr = wn;
                    if (a.c64_lnw && dx < 0x3FA00000u && mid_weight(wn)) {
                        Lk = Lw = log_carry(Lw, Ll, w, wn, d, e);
                    } else {
                        if (a.c64_lnw) { Lk = log(wn / a.what[i]); Ll = 0.0; }
                        Lw = Lw + d;
                    }
                    if (d_bad(wn)) bad = true;
                }
                if (fl & F_STATS) {
                    s_d = fma(-wr, Lw, s_d);
                    w_d += wr;
                }
                if (a.c64_lnw) { a.c64_lnw[i] = Lk; a.c64_lnl[i] = Ll; }
            } else if (__double_as_longlong(w) != 0ll) {
                bad = true;       // negative, -0 or NaN weight
            }
        }
        if (fl & F_PUSH) kdk<double, PK_ANY>(x, y, z, vx, vy, vz, a, sh, i, kept_force<double, PK_ANY>(a, i));
        if (fl & F_SCAT) {
            const double X = x, Ys = z * sn - y * cs, vlos = vy * sn + vz * cs;
            if constexpr (L == 0) {
                for (int k = 0; k < a.nsets; ++k) {
                    const SetDev &s = a.sets[k];
                    double Xk = X, Yk = Ys;
                    if (s.psf) seeing<double>(s, k, i, a.epoch + ((fl & F_PUSH) ? 1 : 0), Xk, Yk);
                    const int c = set_cell<double>(s, S.edges, x, y, z, Xk, Yk);
                    if (c < 0) continue;
                    const int h = (s.obs_off + c * s.nmom) * S.hrep + S.hlane * s.nmom;
                    if (s.quant == M2M_Q_MASS) {
                        hist64(S, h, wn);
                    } else if (s.quant == M2M_Q_VLOS2) {
                        hist64(S, h, wn * (vlos * vlos));
                    } else {
                        double u[5];
                        gh_eval(vlos, S.gh + s.gh_off + 5 * c, u, T);
#pragma unroll
                        for (int m = 0; m < 5; ++m) hist64(S, h + m, wn * u[m]);
                    }
                }
            } else {
                unsigned packed = 0u;
                for_each_set<L>([&](auto K, auto G, auto Q) {
                    constexpr int k = decltype(K)::value, g = decltype(G)::value, q = decltype(Q)::value;
                    const SetDev &s = a.sets[k];
                    const int c = cell64<g>(s, S.ekey, x, y, z, X, Ys);
                    packed |= (unsigned)(c + 1) << s.cshift;
                    if (c < 0) return;
                    if constexpr (q == M2M_Q_MASS) {
                        if (wn != 0.0) hist64(S, (s.obs_off + c) * S.hrep + S.hlane, wn);
                    } else if constexpr (q == M2M_Q_VLOS2) {
                        if (wn != 0.0) hist64(S, (s.obs_off + c) * S.hrep + S.hlane, wn * (vlos * vlos));
                    } else {
                        const double *r = S.gh + s.gh_off + 5 * c;
                        const GhPoint hp = gh_point(r, vlos, T);
                        if (a.c64_m) { a.c64_m[i] = hp.m; a.c64_g[i] = hp.g; }
                        if (wn != 0.0) {
                            // the moments of gh_record's polynomials
                            const double SQ2 = 1.4142135623730951, K3 = 1.1547005383792515, K4 = 0.81649658092772603;
                            const double m = hp.m, m2 = m * m, W = wn * hp.g, d = r[4];
                            const double d4 = d * 2.4494897427831779;               // 12 d/sqrt 24
                            const int h = (s.obs_off + 5 * c) * S.hrep + S.hlane * 5;
                            hist64(S, h, W);
                            hist64(S, h + 1, W * (SQ2 * m));
                            hist64(S, h + 2, W * fma(SQ2, m2, d * 0.70710678118654752));
                            hist64(S, h + 3, W * (m * fma(K3, m2, d * 1.7320508075688772)));
                            hist64(S, h + 4, W * fma(m2, fma(K4, m2, d4), (d * d) * 0.61237243569579447));
                        }
                    }
                });
                if (a.cache_write) a.cell_cache[i] = packed;
            }
        }
        if (fl & F_MINMAX) {
            double E, Lz;
            energy_lz<double, PK_ANY>(x, y, z, vx, vy, vz, a, sh, E, Lz);
            emin = fmin(emin, E);
            emax = fmax(emax, E);
            lzm = fmax(lzm, fabs(Lz));
        }
        if (fl & F_CELLS) {
            const int c = prior_cell<double, PK_ANY>(x, y, z, vx, vy, vz, a, C.pe, C.pl, C.gp, sh);
            a.cell_ids[i] = c;
            cell_add<double>(a, C, c, wn, ovf);
        }
        if (fl & F_PUSH) { px[i] = x; py[i] = y; pz[i] = z; pvx[i] = vx; pvy[i] = vy; pvz[i] = vz; }
        if (fl & F_UPD) a.w[i] = wn;
    }
    if (a.rec_pending) {
        // the record of the preceding step, by the first block to get here
        __shared__ int s_rec;
        if (threadIdx.x == 0) s_rec = atomicAdd(a.rec_ticket, 1ull) == a.rec_base;
        __syncthreads();
        if (s_rec && threadIdx.x < 32)
            record_warp(a.rec_chi, a.rec_chi_nblk, a.rec_stat, a.rec_stat_nblk, a.mu, a.rec_step, a.rec_write_ring,
                        (m2m_record *)a.ring, (m2m_record *)a.last, a.err);
    }
    griddep_launch();
    __syncthreads();
    if (fl & F_SCAT) {
        // the block's sums into the totals; the copies of an observable are
        // at odd strides, so a warp's reads of one copy spread over the banks
        const int R = S.hrep;
        for (int k = threadIdx.x; k < nobs; k += NT) {
            int off = 0, nmom = 1;
            for (int q = 0; q < a.nsets; ++q)
                if (k >= a.sets[q].obs_off) { off = a.sets[q].obs_off; nmom = a.sets[q].nmom; }
            const int m = nmom == 5 ? (k - off) % 5 : 0, base = (k - m) * R + m;
            double v = S.h[base + ((int)threadIdx.x & (R - 1)) * nmom];
            for (int q = 1; q < R; ++q) v += S.h[base + ((q + (int)threadIdx.x) & (R - 1)) * nmom];
            if (v != 0.0) atomicAdd((double *)a.y_acc + k, v);
        }
    }
    if (fl & F_CELLS) {
        for (int k = threadIdx.x; k < a.ncells; k += NT) {
            const unsigned cn = C.c_lo[k];
            if (cn) {
                atomicAdd((double *)a.cell_acc + k, C.c_d[k]);
                atomicAdd(a.cell_cnt + k, cn);
            }
        }
    }
    if (fl & F_STATS) {
        const double s_tot = block_sum(s_d, red), w_tot = block_sum(w_d, red);
        if (threadIdx.x == 0) {
            a.stat_slots[2 * bid] = s_tot;
            a.stat_slots[2 * bid + 1] = w_tot;
        }
    }
    if (fl & F_MINMAX) {
        __shared__ double mm[3][32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            emin = fmin(emin, __shfl_xor_sync(0xffffffffu, emin, o));
            emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
            lzm = fmax(lzm, __shfl_xor_sync(0xffffffffu, lzm, o));
        }
        const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
        if (lane == 0) { mm[0][wp] = emin; mm[1][wp] = emax; mm[2][wp] = lzm; }
        __syncthreads();
        if (threadIdx.x == 0) {
            double e0 = mm[0][0], e1 = mm[1][0], l2 = mm[2][0];
            for (int k = 1; k < NT / 32; ++k) {
                e0 = fmin(e0, mm[0][k]); e1 = fmax(e1, mm[1][k]); l2 = fmax(l2, mm[2][k]);
            }
            double *o = (double *)a.mm_slots + 4 * bid;
            o[0] = e0; o[1] = e1; o[2] = l2; o[3] = 0.0;
        }
    }
    if (ovf) atomicOr(a.err, ERR_OVERFLOW);
    if (bad) atomicOr(a.err, ERR_NONFINITE);
}

template <int NT, int MINB, int L>
__global__ void __launch_bounds__(NT, MINB) k_pass64(const __grid_constant__ PassArgs a) {
    pass64_body<NT, L>(a, blockIdx.x, gridDim.x);
}

}  // namespace m2m
