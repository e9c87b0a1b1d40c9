// Host side of libpaircount: argument checks, the counting plan (stencil,
// lookup tables, FP32 error bands), device workspace, and the count entry
// points pc_count_auto / pc_count_cross / pc_count_batch.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <atomic>
#include <map>
#include <memory>
#include <string>
#include <vector>

#include "pc_host.hpp"

namespace pc {

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
static thread_local std::string g_last_error;

void set_error(const std::string &msg) { g_last_error = msg; }

pc_status fail(pc_status s, const std::string &msg) {
    set_error(msg);
    return s;
}

pc_status cuda_fail(cudaError_t e, const char *what) {
    std::string m = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    set_error(m);
    if (e == cudaErrorMemoryAllocation) return PC_ENOMEM;
    return PC_ECUDA;
}

static std::atomic<long long> g_launches{0};
void note_launch(int n) { g_launches.fetch_add(n); }
long long launch_count() { return g_launches.load(); }

static std::atomic<long long> g_allocs{0};
void note_alloc() { g_allocs.fetch_add(1); }
long long alloc_count() { return g_allocs.load(); }

std::mutex &api_mutex() {
    static std::mutex m;
    return m;
}

bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// ---------------------------------------------------------------------------
// device workspace (grown on demand, reused across calls)
// ---------------------------------------------------------------------------
struct Buf {
    void *p = nullptr;
    size_t cap = 0;
    cudaError_t ensure(size_t bytes) {
        if (bytes <= cap) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
        size_t want = std::max(bytes, cap * 3 / 2);
        cudaError_t e = ::pc::alloc_dev(&p, want);
        if (e != cudaSuccess) {
            cudaGetLastError();
            want = bytes;
            e = ::pc::alloc_dev(&p, want);
        }
        if (e == cudaSuccess) cap = want;
        return e;
    }
};

struct Workspace {
    Buf hist, whist, counters, scalars, queue, blocks, tmp_cnt, tmp_off, tmp_tot, tasks, stencil, lut,
        ea, eb, wsums;
};

// Integer weight products: each of the launch's `grid` CTAs gets its own exact
// sums per bin in the workspace (PairParams::wsums).
static pc_status attach_wsums(Workspace &W, PairParams &p, int grid) {
    if (!p.wint) return PC_OK;
    PC_CUDA(W.wsums.ensure(sizeof(unsigned long long) * 2 * (size_t)p.nbins *
                           (size_t)std::max(grid, 1)));
    p.wsums = (unsigned long long *)W.wsums.p;
    return PC_OK;
}

static Workspace &workspace(int dev) {
    static std::map<int, Workspace> ws;
    return ws[dev];
}

// ---------------------------------------------------------------------------
// plan: bins, error bands, lookup tables, stencil
// ---------------------------------------------------------------------------
struct Plan {
    int mode = 0, los = 0, na = 0, nb = 1, nbins = 0;
    std::vector<double> ea, eb;   // edges
    std::vector<double> Ea, Eb;   // squared edges
    double reff = 0, rcut = 0;
    float eps_a = 0, eps_b = 0, mu_A = 0, mu_B = 0, mu_W = 0;
    std::vector<float2> lut;
    LutDesc la{0, 0, 0.f}, lb{0, 0, 0.f};
    std::vector<int4> stencil;
    float r2cut = 0;
    int fp32_ok = 1;              // error bands usable (else use the FP64 path)
    std::string fp32_why;
    // evenly spaced edges: bins by floor (see PairParams::lin*)
    int lin = 0;
    float lin_invA = 0, lin_offA = 0, lin_thrA = 0, lin_nB = 0, lin_mA = 0, lin_cB = 0;
    int lin_norange = 0, lin_log = 0;
    float lin_invB2 = 0, lin_thrB = 0;
    float lin_offA1 = 0;         // lin_offA + 1, rounded once
    float lin_mS = 0;
    // the pair kernel's choice: tables, or floors from zero, from any edge or
    // of logarithms (the lin fields; also for mu along the midpoint line of
    // sight, which lin leaves out)
    int path = PATH_LUT;
    // fixed-point floors (fix: PATH_FIX*, or 0): scales, the first axis's constant
    // without its band, bands in units of 2^-16 (first axis, fx_sA / s for
    // logarithms; pi of (sigma, pi); mu, fx_mA / s + fx_mB), and the separation the
    // mu band stops growing at
    int fix = 0;
    double fx_c = 128.0, fx_inv = 0, fx_invB = 0, fx_s = 0, fx_sA = 0, fx_p = 0, fx_mA = 0, fx_mB = 0, fx_sf = 0;
};

static bool edges_ok(const double *e, int n, bool zero_one) {
    if (n < 1 || !e) return false;
    for (int k = 0; k <= n; ++k)
        if (!(e[k] >= 0.0) || !isfinite(e[k])) return false;
    for (int k = 0; k < n; ++k)
        if (!(e[k + 1] > e[k])) return false;
    if (zero_one && !(e[0] == 0.0 && e[n] == 1.0)) return false;
    return true;
}

static const double U32 = 5.9604644775390625e-08;   // 2^-24

static float bits_f(int v) {
    float f;
    memcpy(&f, &v, sizeof(f));
    return f;
}

// Lookup table over [0, V): T cells of width V/T, each holding the single
// decision edge within `win` of the cell (or +inf if none, NaN if several)
// and the bin index just below it.  `closed_mu`: the quantity is mu, whose
// first and last edges (0 and 1) are not decisions.
static void build_lut(const std::vector<double> &e, bool closed_mu, double V, double win,
                      std::vector<float2> &out, LutDesc &d) {
    const int n = (int)e.size() - 1;
    std::vector<double> dec;      // decision edges
    std::vector<int> below;       // bin index just below each decision edge
    for (int m = 0; m <= n; ++m) {
        if (closed_mu && (m == 0 || m == n)) continue;
        if (!closed_mu && m == 0 && e[0] == 0.0) continue;   // v >= 0 always holds
        dec.push_back(e[m]);
        below.push_back(m - 1);
    }
    auto bin_of = [&](double v) {   // bin of a value away from every edge
        if (closed_mu) {
            int j = 0;
            for (int m = 1; m < n; ++m) if (v >= e[m]) j = m;
            return j;
        }
        int k = -1;
        for (int m = 0; m <= n; ++m) if (v >= e[m]) k = m;
        return k;   // -1 below e[0], n at or above e[n]
    };
    // smallest table (power of two) whose windows hold at most one edge each
    int T = 16;
    for (; T < MAX_LUT; T *= 2) {
        double w = V / T;
        bool clash = false;
        for (size_t m = 1; m < dec.size() && !clash; ++m)
            if (dec[m] - dec[m - 1] <= w + 2.0 * win) clash = true;
        if (!clash) break;
    }
    float inv_w = (float)(T / V);
    d.off = (int)out.size();
    d.T = T;
    d.inv_w = inv_w;
    const double cw = 1.0 / (double)inv_w;   // actual cell width in value units
    for (int t = 0; t <= T + 1; ++t) {
        float2 ent;
        if (t == T + 1) {   // NaN / inf inputs land here: always rescue
            ent.x = bits_f(0x7fc00000);
            ent.y = bits_f(0);
            out.push_back(ent);
            continue;
        }
        double lo = t * cw - win, hi = (t + 1) * cw + win;
        int cnt = 0, which = -1;
        for (size_t m = 0; m < dec.size(); ++m)
            if (dec[m] >= lo && dec[m] <= hi) { ++cnt; which = (int)m; }
        if (cnt == 0) {
            ent.x = INFINITY;
            int k = bin_of(std::max(0.0, t * cw + 0.5 * cw));
            ent.y = bits_f(k);
        } else if (cnt == 1) {
            ent.x = (float)dec[which];
            ent.y = bits_f(below[which]);
        } else {
            ent.x = bits_f(0x7fc00000);
            ent.y = bits_f(0);
        }
        out.push_back(ent);
    }
}

// Stencil rows (dy, dz, xlo, xhi) of cells whose minimum distance to the
// reference cell is below r (half shell for auto counts, Sect. 3.1).
static void build_stencil(const Geom &g, double r, bool half, std::vector<int4> &rows,
                          int kmax[3]) {
    rows.clear();
    const double slack = 1e-9 * std::max({g.c[0], g.c[1], g.c[2], fabs(g.lo[0]) + g.L[0],
                                           fabs(g.lo[1]) + g.L[1], fabs(g.lo[2]) + g.L[2]});
    auto md = [&](int k, int a) {
        double v = std::max(std::abs(k) - 1, 0) * g.c[a] - 2.0 * slack;
        return v > 0 ? v : 0.0;
    };
    int ky = (int)ceil(r / g.c[1]) + 1, kz = (int)ceil(r / g.c[2]) + 1;
    kmax[0] = kmax[1] = kmax[2] = 0;
    double r2 = r * r;
    for (int dz = -kz; dz <= kz; ++dz) {
        for (int dy = -ky; dy <= ky; ++dy) {
            double m2 = md(dy, 1) * md(dy, 1) + md(dz, 2) * md(dz, 2);
            if (m2 >= r2) continue;
            int rx = 0;
            while (true) {
                double mx = md(rx + 1, 0);
                if (mx * mx + m2 < r2) ++rx; else break;
            }
            int xlo = -rx, xhi = rx;
            if (half) {
                // Sect. 3.1 duplicate removal: of every row pair (dy, dz),
                // (-dy, -dz) exactly one is visited.  The kept member alternates
                // with the parity of dy + dz (the parity is the same for both),
                // so the visited half reaches equally far up and down: every
                // warp's i-points then see the same volume wherever they sit in
                // the cell, and the warps of a CTA stay balanced.
                if (dz == 0 && dy == 0) {
                    if (rx < 1) continue;
                    xlo = 1;
                } else {
                    const bool upper = dz > 0 || (dz == 0 && dy > 0);
                    if (upper == (((dy + dz) & 1) != 0)) continue;
                }
            }
            rows.push_back(make_int4(dy, dz, xlo, xhi));
            kmax[0] = std::max(kmax[0], rx);
            kmax[1] = std::max(kmax[1], std::abs(dy));
            kmax[2] = std::max(kmax[2], std::abs(dz));
        }
    }
}

static pc_status make_plan(const pc_bins *b, const Geom &g, const double *pts_lo,
                           const double *pts_hi, double rmin, bool half, Plan &P,
                           bool with_stencil = true) {
    if (!b) return fail(PC_EINVAL, "bins: NULL");
    if (b->mode < 0 || b->mode > 2) return fail(PC_EINVAL, "bins: unknown mode");
    if (b->los < 0 || b->los > 1) return fail(PC_EINVAL, "bins: unknown line of sight");
    P.mode = b->mode;
    P.los = (b->mode == PC_BIN_S) ? PC_LOS_Z : b->los;
    if (!edges_ok(b->edges_a, b->n_a, false))
        return fail(PC_EINVAL, "bins: edges_a must be finite, >= 0 and strictly increasing");
    P.na = b->n_a;
    P.ea.assign(b->edges_a, b->edges_a + b->n_a + 1);
    if (P.mode == PC_BIN_S) {
        P.nb = 1;
        P.eb = {0.0, 1.0};
    } else {
        if (!edges_ok(b->edges_b, b->n_b, P.mode == PC_BIN_SMU))
            return fail(PC_EINVAL, P.mode == PC_BIN_SMU
                                       ? "bins: mu edges must increase strictly from 0 to 1"
                                       : "bins: pi edges must be finite, >= 0 and increasing");
        P.nb = b->n_b;
        P.eb.assign(b->edges_b, b->edges_b + b->n_b + 1);
    }
    if ((long long)P.na * P.nb > (1LL << 26)) return fail(PC_EOVERFLOW, "bins: too many bins");
    P.nbins = P.na * P.nb;
    if (g.periodic && P.los == PC_LOS_MIDPOINT)
        return fail(PC_EINVAL, "bins: the midpoint line of sight needs a non-periodic box");
    P.Ea.resize(P.na + 1);
    P.Eb.resize(P.nb + 1);
    for (int k = 0; k <= P.na; ++k) P.Ea[k] = P.ea[k] * P.ea[k];
    for (int k = 0; k <= P.nb; ++k) P.Eb[k] = P.eb[k] * P.eb[k];
    P.reff = (P.mode == PC_BIN_SIGPI) ? sqrt(P.ea[P.na] * P.ea[P.na] + P.eb[P.nb] * P.eb[P.nb])
                                      : P.ea[P.na];

    // ---- FP32 error bands (derivation in the design notes) -----------------
    const double u = U32;
    const double c = std::max({g.c[0], g.c[1], g.c[2]});
    double X = 0.0, Lm = 0.0;
    for (int a = 0; a < 3; ++a) {
        X = std::max({X, fabs(pts_lo[a]), fabs(pts_hi[a])});
        Lm = std::max(Lm, g.L[a]);
    }
    const double R0 = P.reff;
    const double tiny = ldexp(X + Lm + R0, -48);
    // separation length s (and sigma along z) and the z component
    double Rb = R0 * (1.0 + 1e-6) + 1e-6 * c;
    double eps_s = 2.0 * u * (4.4 * c + 10.5 * Rb) + tiny;
    double eps_z = 2.0 * u * (2.5 * c + 4.0 * Rb) + tiny;
    double eps_sig = 2.0 * u * (3.6 * c + 11.5 * Rb) + ldexp(Rb, -25) + tiny;
    double muA = 2.0 * (6.9 * u * c) + tiny, muB = 2.0 * 21.0 * u + ldexp(1.0, -48);
    double lmin = 0.0;   // midpoint: lower bound of |x_i + x_j|
    if (P.los == PC_LOS_MIDPOINT) {
        // distance of the nearest point to the observer bounds |x_i + x_j|:
        // the larger of the bounding box's distance and the points' own
        // smallest radius (a shell is far from the observer although its
        // bounding box may come close)
        double dmin2 = 0.0;
        for (int a = 0; a < 3; ++a) {
            double d = 0.0;
            if (pts_lo[a] > 0.0) d = pts_lo[a];
            else if (pts_hi[a] < 0.0) d = -pts_hi[a];
            dmin2 += d * d;
        }
        const double dmin = std::max(sqrt(dmin2) * (1.0 - 1e-12), rmin);
        lmin = 2.0 * dmin - Rb;
        double dl = u * (5.5 * X + 4.4 * c + 6.2 * Rb);
        if (lmin > 4.0 * Rb) {
            double em = 2.0 * (u * (4.4 * c + 17.5 * Rb) + 2.0 * Rb * dl / lmin) +
                        ldexp(Rb, -25) + tiny;
            eps_sig = em;
            eps_z = em;
            muA = em + eps_s;
            muB = 2.0 * 8.0 * u + ldexp(1.0, -48);
        } else {
            P.fp32_ok = 0;
            P.fp32_why = "observer too close to the points for the FP32 midpoint bound";
        }
    }
    P.rcut = R0 + std::max({eps_s, eps_z, eps_sig}) * 2.0;
    // binary32 squares of separations in range (midpoint: and of x_i + x_j) must be
    // finite, or pairs were lost: a box of 2^60 x 100 with reach 2^60 x 30 kept 15 % of
    // its pairs, one of 2^66 none
    if (!(P.rcut < 1.7e19) || (P.los == PC_LOS_MIDPOINT && !(4.0 * X + R0 < 1.7e19))) {
        P.fp32_ok = 0;
        P.fp32_why = "binary32 squares of the separations overflow";
    }
    {
        double r2 = P.rcut * P.rcut * (1.0 + 8.0 * u);
        P.r2cut = nextafterf((float)r2, INFINITY);
    }
    // ---- lookup tables ------------------------------------------------------
    const double V = P.rcut * (1.0 + 1e-5) + 1e-30;
    P.lut.clear();
    if (P.mode == PC_BIN_S) {
        P.eps_a = (float)(eps_s * (1.0 + 1e-6));
        build_lut(P.ea, false, V, 2.0 * eps_s, P.lut, P.la);
        P.lb = P.la;
    } else if (P.mode == PC_BIN_SMU) {
        P.eps_a = (float)(eps_s * (1.0 + 1e-6));
        P.mu_A = (float)(muA * (1.0 + 1e-6));
        P.mu_B = (float)(muB * (1.0 + 1e-6));
        build_lut(P.ea, false, V, 2.0 * eps_s, P.lut, P.la);
        // mu window: the band of a pair must fit in it (else always rescue)
        double minGap = 1.0;
        for (int k = 0; k < P.nb; ++k) minGap = std::min(minGap, P.eb[k + 1] - P.eb[k]);
        double wmu = std::min(1e-3, 0.2 * minGap);
        P.mu_W = (float)wmu;
        build_lut(P.eb, true, 1.0 + 1e-3, wmu, P.lut, P.lb);
    } else {
        P.eps_a = (float)(eps_sig * (1.0 + 1e-6));
        P.eps_b = (float)(eps_z * (1.0 + 1e-6));
        build_lut(P.ea, false, V, 2.0 * eps_sig, P.lut, P.la);
        build_lut(P.eb, false, V, 2.0 * eps_z, P.lut, P.lb);
    }
    // mu floors along the midpoint line of sight run only inside the kernel's
    // own choice (P.path); the lin view stays with the z line of sight
    const bool mid_mu = P.mode == PC_BIN_SMU && P.los == PC_LOS_MIDPOINT;
    // mu = |d.l| rsqrt(l^2) rsqrt(s^2) may exceed 1 by rounding: along z by the
    // reciprocal root's and the squares' errors (3e-7), along the midpoint by
    // 12.3 u = 7.4e-7 (3 u from d.l, 1.5 u from each square, 2.15 u from each
    // reciprocal root, 2 u from the products); the scale stays below n_mu by more
    const double mu_shrink = ldexp(1.0, mid_mu ? -20 : -21);
    // ---- evenly spaced edges: floor-based bins ------------------------------
    // s (and mu along z): bin = floor(t), t = (s - e0) / D, with the band
    // moved into t units plus the rounding of t itself (scaling factor and
    // offset rounded to FP32, one FMA) and the edges' distance from exact
    // even spacing.
    {
        const double e0 = P.ea[0], D = (P.ea[P.na] - P.ea[0]) / P.na;
        double dev = 0.0;
        for (int k = 0; k <= P.na; ++k) dev = std::max(dev, fabs(P.ea[k] - (e0 + k * D)));
        bool lin_s = dev <= 1e-9 * D;
        bool lin_mu = true;
        double devm = 0.0;
        if (P.mode == PC_BIN_SMU) {
            for (int k = 0; k <= P.nb; ++k) devm = std::max(devm, fabs(P.eb[k] - (double)k / P.nb));
            lin_mu = (P.los == PC_LOS_Z || P.fp32_ok) && devm <= 1e-12;
        }
        bool mode_ok = P.mode == PC_BIN_S || P.mode == PC_BIN_SMU;
        if (lin_s && lin_mu && mode_ok && (P.rcut - e0) / D < 4.0e6) {
            double ts_max = (P.rcut - e0) / D + 1.0;
            double eps_t = (eps_s + dev) / D + 4.0 * u * (ts_max + fabs(e0) / D);
            if (eps_t < 0.25) {
                P.lin = 1;
                P.lin_invA = (float)(1.0 / D);
                P.lin_offA = (float)(-e0 / D);
                P.lin_offA1 = (float)(1.0 - e0 / D);
                P.lin_thrA = nextafterf((float)(0.5 - eps_t), 0.0f);
                // e_0 = 0: t_s = s / D >= 0; and every candidate has t_s below
                // n_a + 1/2 (plus rounding), so floor(t_s) <= n_a
                P.lin_norange = (e0 == 0.0 && ts_max - 1.0 <= P.na + 0.5) ? 1 : 0;
                if (P.mode == PC_BIN_SMU) {
                    // t_mu = mu n_mu (1 - 2^-21): below n_mu for every pair (mu
                    // = |dz| rsqrt(s^2) exceeds 1 by at most ~3e-7), so mu = 1
                    // lands in the last bin without a clamp; the scale's shift
                    // of up to 2^-21 n_mu joins the band
                    const double nb = P.nb;
                    P.lin_nB = nextafterf((float)(nb * (1.0 - mu_shrink)), 0.0f);
                    P.lin_mA = (float)(muA * nb * (1.0 + 1e-6));
                    double cB = 0.5 - (muB + 4.0 * u + devm + mu_shrink) * nb;
                    P.lin_cB = nextafterf((float)cB, 0.0f);
                    if (!(cB > 0.25)) P.lin = 0;
                }
            }
        }
    }
    // ---- logarithmic s edges: floor of a scaled base-2 logarithm -----------
    // e_k = e_0 q^k: bin = floor(t), t = log_q(s / e_0) = A log2(s^2) + B with
    // A = 1 / (2 log2 q), B = -log2(e_0) / log2 q (Sect. 3.2's log mapping).
    // Band in t units (each term times 2 below, like the linear case):
    //  - the separation vector's error u (4.33 c + 3 s) + 2^-51 X (c the cell
    //    side) is relative in log2(s^2): 2 (4.33 u c + 2^-51 X) / (s ln 2) plus
    //    6u / ln 2, and the three roundings of s^2 add 3u / ln 2 -- the 1/s
    //    part is applied per pair through rsqrt(s^2);
    //  - the hardware base-2 logarithm errs by at most 2^-21 max(1, |log2 x|)
    //    (twice the largest error over every positive normal binary32 input,
    //    measured exhaustively on the device by the test suite);
    //  - A, B rounded to binary32 and the FMA add u (A |L| + |B| + |t|);
    //  - the edges' distance from an exact geometric sequence (in t units),
    //    and the oracle's binary64 roundings (2^-45 A).
    if (!P.lin && P.ea[0] > 0.0) {
        const double e0 = P.ea[0], lq = log2(P.ea[P.na] / e0) / P.na;
        bool lin_mu = true;
        double devm = 0.0;
        if (P.mode == PC_BIN_SMU) {
            for (int k = 0; k <= P.nb; ++k) devm = std::max(devm, fabs(P.eb[k] - (double)k / P.nb));
            lin_mu = (P.los == PC_LOS_Z || P.fp32_ok) && devm <= 1e-12;
        }
        bool mode_ok = P.mode == PC_BIN_S || P.mode == PC_BIN_SMU;
        double dev = 0.0;
        for (int k = 0; k <= P.na; ++k) dev = std::max(dev, fabs(log2(P.ea[k] / e0) / lq - k));
        if (mode_ok && lin_mu && lq > 0.0 && dev <= 1e-6 && P.na < (1 << 20)) {
            const double ln2 = log(2.0), A = 1.0 / (2.0 * lq), B = -log2(e0) / lq;
            const double Lmax = std::max(fabs(log2(P.rcut * P.rcut)), fabs(log2(0.25 * e0 * e0)));
            const double tmax = A * Lmax + fabs(B) + 1.0;
            const double C1 = A * 2.0 * (4.4 * u * c + ldexp(X + Lm + R0, -51)) / ln2 * 1.01;
            const double C0 = A * 9.0 * u / ln2 * 1.01 + A * ldexp(1.0, -21) * std::max(1.0, Lmax) +
                              u * (A * Lmax + fabs(B) + tmax) * 2.0 + dev + A * ldexp(1.0, -45);
            if (2.0 * C0 < 0.25) {
                P.lin = 1;
                P.lin_log = 1;
                P.lin_invA = (float)A;
                P.lin_offA = (float)B;
                P.lin_offA1 = (float)(B + 1.0);
                P.lin_thrA = nextafterf((float)(0.5 - 2.0 * C0), 0.0f);
                // rsqrt(s^2) >= (1 - 2^-22) / s: scale the 1/s term up to cover it
                P.lin_mS = nextafterf((float)(2.0 * C1 * (1.0 + 1e-6)), INFINITY);
                P.lin_norange = 0;
                if (P.mode == PC_BIN_SMU) {
                    const double nb = P.nb;   // mu scale and band as for linear s bins
                    P.lin_nB = nextafterf((float)(nb * (1.0 - mu_shrink)), 0.0f);
                    P.lin_mA = (float)(muA * nb * (1.0 + 1e-6));
                    double cB = 0.5 - (muB + 4.0 * u + devm + mu_shrink) * nb;
                    P.lin_cB = nextafterf((float)cB, 0.0f);
                    if (!(cB > 0.25)) P.lin = P.lin_log = 0;
                }
            }
        }
    }
    P.path = !P.lin ? PATH_LUT : (P.lin_log ? PATH_LOG : (P.ea[0] == 0.0 ? PATH_LIN : PATH_LINOFF));
    if (mid_mu) P.lin = P.lin_log = P.lin_norange = 0;
    // ---- (sigma, pi) with evenly spaced edges from 0: floors of both ------
    // t_sigma = sigma / D_a, t_pi = pi / D_b, sigma and pi formed as on the
    // table path, so their bands eps_sig and eps_z apply (in t units), plus
    // the rounding of the scale and product (2u t) and the edges' distance
    // from even spacing.
    if (!P.lin && P.mode == PC_BIN_SIGPI && P.fp32_ok && P.ea[0] == 0.0 && P.eb[0] == 0.0) {
        const double Da = P.ea[P.na] / P.na, Db = P.eb[P.nb] / P.nb;
        double deva = 0.0, devb = 0.0;
        for (int k = 0; k <= P.na; ++k) deva = std::max(deva, fabs(P.ea[k] - k * Da));
        for (int k = 0; k <= P.nb; ++k) devb = std::max(devb, fabs(P.eb[k] - k * Db));
        const double tma = P.rcut / Da + 1.0, tmb = P.rcut / Db + 1.0;
        const double eta = (eps_sig + deva) / Da + 4.0 * u * tma;
        const double etb = (eps_z + devb) / Db + 4.0 * u * tmb;
        if (deva <= 1e-9 * Da && devb <= 1e-9 * Db && tma < 4.0e6 && tmb < 4.0e6 && eta < 0.25 &&
            etb < 0.25) {
            P.lin = 1;
            P.lin_invA = (float)(1.0 / Da);
            P.lin_offA = 0.0f;
            P.lin_offA1 = 0.0f;
            P.lin_thrA = nextafterf((float)(0.5 - eta), 0.0f);
            P.lin_invB2 = (float)(1.0 / Db);
            P.lin_thrB = nextafterf((float)(0.5 - etb), 0.0f);
            P.lin_norange = 0;
            P.path = PATH_LIN;
        }
    }
    // ---- fixed-point floors (PATH_FIX*) ---------------------------------------
    // The values of the floors, summed once onto a grid of 2^-16: the band in
    // these units, with half a unit for that sum (and with an offset another for
    // the constant's rounding, below 256).  Along z the linear bounds above are
    // used with a factor of 1.25 instead of 2: per axis u (2.5 c + 3 |d|), hence s
    // errs by u (4.33 c + 3 s), the squares' roundings add 1.5 u s, the reciprocal
    // root 2.15 u s, and the scale and its product 2 u s (the last product is
    // exact); mu by u (6.83 c / s + 3 + 3 + 1.5 + 2.15 + 1).
    {
        const double one = 65536.0;
        const double na = P.na, nb = P.nb;
        int kind = P.path == PATH_LIN ? PATH_FIX : (P.path == PATH_LINOFF ? PATH_FIXOFF
                                                    : (P.path == PATH_LOG ? PATH_FIXLOG : 0));
        const double D = (P.ea[P.na] - P.ea[0]) / na;
        bool ok = true;
        // edges evenly spaced from zero (second axis of (sigma, pi)), and
        // logarithmic sigma edges: dt = d sigma / (sigma ln q), sigma >= e_0 / 2
        double Db = D, lq = 0.0;
        if (P.mode == PC_BIN_SIGPI) {
            Db = P.eb[P.nb] / nb;
            double devb = 0.0;
            for (int k = 0; k <= P.nb; ++k) devb = std::max(devb, fabs(P.eb[k] - k * Db));
            if (!kind && P.fp32_ok && P.ea[0] > 0.0 && P.eb[0] == 0.0 && devb <= 1e-9 * Db) {
                lq = log2(P.ea[P.na] / P.ea[0]) / na;
                double dev = 0.0;
                for (int k = 0; k <= P.na; ++k) dev = std::max(dev, fabs(log2(P.ea[k] / P.ea[0]) / lq - k));
                if (dev <= 1e-6 && eps_sig < 0.05 * P.ea[0]) kind = PATH_FIXLOG;
            }
            P.fx_invB = 1.0 / Db;
            P.fx_p = ceil((eps_z / Db + 1e-9 + 4.0 * u * nb) * one + 0.5);
            ok = ok && P.fx_p < 8192.0;
        }
        if (kind == PATH_FIXLOG) {
            const double e0 = P.ea[0];
            if (lq == 0.0) lq = log2(P.ea[P.na] / e0) / na;
            const double ln2 = log(2.0), A = 1.0 / (2.0 * lq), B = -log2(e0) / lq;
            const double Lmax = std::max(fabs(log2(P.rcut * P.rcut)), fabs(log2(0.25 * e0 * e0)));
            const double common = A * ldexp(1.0, -21) * std::max(1.0, Lmax) +
                                  u * (A * Lmax + fabs(B) + na + 130.0) * 2.0 + 1e-6 + A * ldexp(1.0, -45);
            P.fx_inv = A;
            P.fx_c = 129.0 + B;
            if (P.mode == PC_BIN_SIGPI) {
                P.fx_sA = 1.12 * eps_sig / (lq * ln2) * one;
                P.fx_s = 2.0 * common * one + 2.0;
            } else {
                P.fx_sA = 2.0 * A * 2.0 * (4.4 * u * c + ldexp(X + Lm + R0, -51)) / ln2 * 1.01 * one;
                P.fx_s = 2.0 * (A * 9.0 * u / ln2 * 1.01 + common) * one + 2.0;
            }
            P.fx_sA *= 1.001;
            ok = ok && e0 > 1e-9 && eps_s < 0.05 * e0 && fabs(P.fx_c) < 250.0 && P.fx_sA / (0.5 * e0) + P.fx_s < 8192.0 && na < FIX_TOP;
        } else if (kind) {
            const double es = P.mode == PC_BIN_SIGPI
                                  ? eps_sig / D + 1e-9 + 4.0 * u * na
                                  : (1.25 * u * (4.34 * c + 8.7 * Rb) + tiny) / D + 1e-9;
            P.fx_inv = 1.0 / D;
            P.fx_c = kind == PATH_FIX ? 128.0 : 129.0 - P.ea[0] / D;
            P.fx_s = ceil(es * one + (kind == PATH_FIX ? 0.5 : 1.5));
            ok = ok && P.fx_s < 8192.0 && (kind == PATH_FIX || (na < FIX_TOP && fabs(P.fx_c) < 250.0));
        }
        if (P.mode == PC_BIN_SMU) {
            const double mA = P.los == PC_LOS_Z ? 1.25 * 6.9 * u * c + tiny : muA;
            const double mB = P.los == PC_LOS_Z ? 1.25 * 10.7 * u + ldexp(1.0, -46) : muB + 4.0 * u;
            P.fx_invB = nb;   // mu = 1 may land in column n_mu: near, put right there
            // Pairs closer than this are near whatever their mu, and batches whose boxes
            // touch take the band there.  c / 16 suits catalogues with few such pairs and
            // many mu bins.  With fewer bins the band allows less, down to c / 64, until it
            // is 1/2048 of a bin, which spares tight clusters (c / 16 found half of a
            // cluster's pairs near; 1/512 cost cross counts of 40 bins 5 to 12 %), and in
            // cells or list nodes above twice the reach it is an eighth of the reach (at a
            // reach of 5 every pair of a 250-point node was closer than c / 16)
            P.fx_sf = std::max(std::min({c / 16.0, R0 / 8.0, std::max(c / 64.0, 2048.0 * nb * mA)}), 1e-3 * R0);
            P.fx_mA = nb * mA * one * 1.001;
            P.fx_mB = nb * mB * one * 1.001 + 1e-12 * nb * one + 1.0;
            ok = ok && P.fx_mA / P.fx_sf + P.fx_mB < 8192.0;
        }
        // no FP32 square may overflow (the kernel's indices rely on it), and the
        // constant 1e-30 in the squares must stay far inside the first band
        ok = ok && X + Lm + R0 + c < 1e15 && std::min({D, Db, P.ea[1]}) > 1e-9 && na <= FIX_TOP && nb <= FIX_TOP;
        // along the midpoint |d x l|^2 is a fourth power (|l| <= 2 sqrt(3) X): it comes to
        // the ends of binary32 and near that constant first, in units far from a
        // catalogue's scale (limits of a survey shell in Mpc: times 2^21 and 2^-21);
        // packed floors and tables find such pairs near an edge
        if (P.mode == PC_BIN_SIGPI && P.los == PC_LOS_MIDPOINT)
            ok = ok && R0 * (4.0 * X + R0) < 1.7e19 && (P.ea[0] > 0.0 ? P.ea[0] : P.ea[1]) * lmin > 1e-9;
        P.fix = ok ? kind : 0;
    }
    // ---- stencil -------------------------------------------------------------
    int kmax[3] = {0, 0, 0};
    P.stencil.clear();
    if (with_stencil) build_stencil(g, P.rcut, half, P.stencil, kmax);
    if (g.periodic) {
        for (int a = 0; a < 3; ++a) {
            if (!(P.rcut < 0.5 * g.L[a]))
                return fail(PC_EINVAL,
                            "bins: the largest separation must stay below half the periodic box");
            if (with_stencil && 2 * kmax[a] + 1 > g.ng[a])
                return fail(PC_EINVAL,
                            "grid: cells too large for this separation in a periodic box "
                            "(neighbour cells would alias); rebuild with a smaller cell_size");
        }
    }
    return PC_OK;
}

// ---------------------------------------------------------------------------
// one counting launch over a set of tasks
// ---------------------------------------------------------------------------
// Histogram replication from pc_opts.priv: 2 = a single shared copy,
// otherwise lane copies (lane l updates copy l % k), as many as fit a 16 KB
// budget, so the lanes of a warp do not collide on the few bins of a small
// histogram (1 also keeps the weighted sums in binary64).
// (weighted: binary64 weight sums share the copies and the budget; the
// integer weight records take the counts' copies outside that budget.)
static void choose_replication(int mode, int nbins, bool weighted, int &hist_k) {
    hist_k = 1;
    if (mode == 2) return;
    const long long per_copy = (long long)nbins * (4 + (weighted ? 8 : 0));
    while (hist_k < 32 && per_copy * hist_k * 2 <= 16384) hist_k *= 2;
}

// Entries of each shared histogram copy: rows of hs entries and one discarded
// entry past them.  The (sigma, pi) floors send pi past its last bin to a
// discarded column.
static void set_hist_rows(PairParams &p, const Plan &P) {
    p.hs = P.nb + (P.mode == PC_BIN_SIGPI && p.path == PATH_LIN ? 1 : 0);
    p.nent = P.na * p.hs + 1;
}

struct CountJob {
    std::vector<TaskDev> tasks;
    int nhist;
    bool is_auto;
    const pc_grid *g0 = nullptr;
    // geometry of the count (the first grid's, or the trees')
    Geom geom;
    int device = 0;
    int ncell = 0;               // cells per grid, or i-blocks of a tree count
    double plo[3] = {0, 0, 0}, phi[3] = {0, 0, 0};   // first grid's point bounds
    double cell_size = 0.0;
    bool tree = false;
    // bounds of the points of every grid involved, and a lower bound of |x|
    double lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
    double rmin = 0.0;
    bool wint_ok = true;   // every task's grids allow the integer weight path
    bool wcorr = false;    // some grid's binary64 weights add remainders
};

// Integer weight products are truncated by at most 2^(k_i + k_j - 46)
// relative, k the exponent offset of a weight below its grid's largest; the
// exponent spans of the two grids are limited so that this stays below
// 2^-34 (6e-11) per product and hence per bin.
static void job_add_wint(CountJob &J, const pc_grid *gi, const pc_grid *gj) {
    if (!gi->wint || !gj->wint ||
        (gi->wemax - gi->wemin) + (gj->wemax - gj->wemin) > WINT_MAX_SPAN)
        J.wint_ok = false;
    if (gi->wcorr || gj->wcorr) J.wcorr = true;
}

// Lower bound of |x| over the points of a grid (0 when unknown or periodic).
static double grid_rmin(const pc_grid *g) {
    if (g->g.periodic || !(g->r2min > 0.0)) return 0.0;
    return sqrt(g->r2min) * (1.0 - 1e-12);
}

// The job's geometry from its first grid.
static void job_set_grid(CountJob &J, const pc_grid *g) {
    J.g0 = g;
    J.geom = g->g;
    J.device = g->device;
    J.ncell = g->ncell;
    for (int a = 0; a < 3; ++a) {
        J.plo[a] = g->pts_lo[a];
        J.phi[a] = g->pts_hi[a];
    }
    J.cell_size = g->cell_size;
}

// Fold grid g into the job's point bounds (the first grid initialises them).
static void job_add_bounds(CountJob &J, const pc_grid *g, bool first) {
    for (int a = 0; a < 3; ++a) {
        J.lo[a] = first ? g->pts_lo[a] : std::min(J.lo[a], g->pts_lo[a]);
        J.hi[a] = first ? g->pts_hi[a] : std::max(J.hi[a], g->pts_hi[a]);
    }
    J.rmin = first ? grid_rmin(g) : std::min(J.rmin, grid_rmin(g));
}

// Everything decided on the host before any device work.
struct CountSetup {
    Plan P;
    pc_opts o;
    int prec = 0, ipt = 2, bi = 256, dev = 0, ntasks = 0, ncell = 0;
    bool weighted = false;
    int wsum = 0;   // weighted sums: 0 none, 1 binary64 products, 2 integer products,
                    // 3 integer products with binary64 remainders
    size_t nblk_cap = 0, hist_n = 0;
    unsigned long long qcap = 0;
};

// Device buffers of one count (raw pointers into a Workspace).
struct DevBufs {
    unsigned long long *hist = nullptr;
    double *whist = nullptr;
    unsigned long long *ctr = nullptr;   // [0] candidates, [1] inline rescues, [2] queue count,
                                         // [3] pairs pruned by the octs' boxes
    int *sc = nullptr;                   // [0] work counter, [1] number of blocks
    uint3 *queue = nullptr;
    Block *blocks = nullptr;
    int *cnt = nullptr, *off = nullptr, *tot = nullptr;
    TaskDev *tasks = nullptr;
    int4 *stencil = nullptr;
    float2 *lut = nullptr;
    double *ea = nullptr, *eb = nullptr;
};

static pc_status setup_count(const CountJob &J, const pc_bins *b, const pc_opts *opt,
                             bool weighted, CountSetup &S) {
    memset(&S.o, 0, sizeof(S.o));
    S.o.priv = -1;
    if (opt) S.o = *opt;
    if (S.o.shard_count > 1 && (S.o.shard_index < 0 || S.o.shard_index >= S.o.shard_count))
        return fail(PC_EINVAL, "opts: shard_index must lie in [0, shard_count)");
    pc_status s = make_plan(b, J.geom, J.lo, J.hi, J.rmin, J.is_auto, S.P, !J.tree);
    if (s != PC_OK) return s;
    S.weighted = weighted;
    S.prec = S.o.prec;
    if (S.prec == PC_PREC_F32_RESCUE && !S.P.fp32_ok) S.prec = PC_PREC_F64;
    S.ipt = (S.o.ipt == 4) ? 4 : 2;
    if (S.prec == PC_PREC_F64) S.ipt = 1;
    S.bi = NT * S.ipt;
    S.dev = J.device;
    S.ntasks = (int)J.tasks.size();
    S.ncell = J.ncell;
    long long npts = 0;
    for (auto &t : J.tasks) npts += t.gi.n;
    S.nblk_cap = (size_t)S.ntasks * S.ncell + (size_t)(npts / S.bi) + 16;
    S.hist_n = (size_t)J.nhist * S.P.nbins;
    // rescue queue: only when asked for.  Near-edge pairs are checked inside
    // the pair kernel otherwise, where their binary64 work overlaps the FP32
    // pairs of the other warps
    S.qcap = 0;
    if (S.prec == PC_PREC_F32_RESCUE) {
        if (S.o.rescue_capacity > 0) S.qcap = (unsigned long long)S.o.rescue_capacity;
    }
    return PC_OK;
}

static pc_status ensure_bufs(Workspace &W, const CountSetup &S, DevBufs &B) {
    const size_t cells = (size_t)S.ntasks * S.ncell + 1;
    PC_CUDA(W.hist.ensure(sizeof(unsigned long long) * S.hist_n));
    if (S.weighted) PC_CUDA(W.whist.ensure(sizeof(double) * S.hist_n));
    PC_CUDA(W.counters.ensure(sizeof(unsigned long long) * 4));
    PC_CUDA(W.scalars.ensure(sizeof(int) * 4));
    PC_CUDA(W.blocks.ensure(sizeof(Block) * S.nblk_cap));
    PC_CUDA(W.tmp_cnt.ensure(sizeof(int) * cells));
    PC_CUDA(W.tmp_off.ensure(sizeof(int) * cells));
    PC_CUDA(W.tmp_tot.ensure(sizeof(int) * (cells / 4096 + 2)));
    PC_CUDA(W.tasks.ensure(sizeof(TaskDev) * S.ntasks));
    PC_CUDA(W.stencil.ensure(sizeof(int4) * std::max<size_t>(S.P.stencil.size(), 1)));
    PC_CUDA(W.lut.ensure(sizeof(float2) * std::max<size_t>(S.P.lut.size(), 1)));
    PC_CUDA(W.ea.ensure(sizeof(double) * (S.P.na + 1)));
    PC_CUDA(W.eb.ensure(sizeof(double) * (S.P.nb + 1)));
    if (S.qcap) PC_CUDA(W.queue.ensure(sizeof(uint3) * S.qcap));
    B.hist = (unsigned long long *)W.hist.p;
    B.whist = S.weighted ? (double *)W.whist.p : nullptr;
    B.ctr = (unsigned long long *)W.counters.p;
    B.sc = (int *)W.scalars.p;
    B.queue = (uint3 *)W.queue.p;
    B.blocks = (Block *)W.blocks.p;
    B.cnt = (int *)W.tmp_cnt.p;
    B.off = (int *)W.tmp_off.p;
    B.tot = (int *)W.tmp_tot.p;
    B.tasks = (TaskDev *)W.tasks.p;
    B.stencil = (int4 *)W.stencil.p;
    B.lut = (float2 *)W.lut.p;
    B.ea = (double *)W.ea.p;
    B.eb = (double *)W.eb.p;
    return PC_OK;
}

// Host-built tables of the count (tasks, stencil, lookup tables, edges).
static pc_status upload_tables(const CountJob &J, const CountSetup &S, const DevBufs &B,
                               cudaStream_t st) {
    PC_CUDA(cudaMemcpyAsync(B.tasks, J.tasks.data(), sizeof(TaskDev) * S.ntasks,
                            cudaMemcpyHostToDevice, st));
    if (!S.P.stencil.empty())
        PC_CUDA(cudaMemcpyAsync(B.stencil, S.P.stencil.data(), sizeof(int4) * S.P.stencil.size(),
                                cudaMemcpyHostToDevice, st));
    if (!S.P.lut.empty())
        PC_CUDA(cudaMemcpyAsync(B.lut, S.P.lut.data(), sizeof(float2) * S.P.lut.size(),
                                cudaMemcpyHostToDevice, st));
    PC_CUDA(cudaMemcpyAsync(B.ea, S.P.Ea.data(), sizeof(double) * (S.P.na + 1),
                            cudaMemcpyHostToDevice, st));
    PC_CUDA(cudaMemcpyAsync(B.eb, S.P.Eb.data(), sizeof(double) * (S.P.nb + 1),
                            cudaMemcpyHostToDevice, st));
    return PC_OK;
}

// The FP32 path's constants from the plan, and the box tests' limits.
static void set_fp32_params(const Geom &g, const double *lo, const double *hi, const Plan &P, int prec,
                            PairParams &p) {
    p.path = (prec == PC_PREC_F32_RESCUE) ? P.path : PATH_LUT;
    p.lin_invA = P.lin_invA;
    // the floors with an offset take t_s + 1 (exact floors down to t_s = -1)
    p.lin_offA = P.lin_offA1;
    p.lin_thrA = P.lin_thrA;
    p.lin_mS = P.lin_mS;
    p.lin_nB = P.lin_nB;
    p.lin_mA = P.lin_mA;
    p.lin_cB = P.lin_cB;
    p.lin_invB2 = P.lin_invB2;
    p.lin_thrB = P.lin_thrB;
    set_hist_rows(p, P);
    {
        auto two = [](float v) { return make_float2(v, v); };
        const double one = 65536.0;
        p.fix = prec == PC_PREC_F32_RESCUE ? P.fix : 0;
        p.row0 = 0;
        const bool off = P.fix == PATH_FIXOFF || P.fix == PATH_FIXLOG;
        p.f_inv = (float)P.fx_inv;
        p.f_invB = (float)P.fx_invB;
        p.f_tiny = two(1e-30f);
        p.f_cfs = two((float)(P.fx_c + (P.fix == PATH_FIXLOG ? 0.0 : P.fx_s / one)));
        p.f_ts2 = 2 * (unsigned)ceil(P.fx_s);
        p.f_cfp = (float)(128.0 + P.fx_p / one);
        p.f_tp2 = 2 * (unsigned)P.fx_p;
        p.f_lim = (off ? 129.5f : 128.5f) + (float)P.na;
        p.f_limB = 128.5f + (float)P.nb;
        p.f_mA = nextafterf((float)P.fx_mA, INFINITY);
        p.f_mB = nextafterf((float)P.fx_mB, INFINITY);
        p.f_sA = nextafterf((float)P.fx_sA, INFINITY);
        p.f_sC = nextafterf((float)P.fx_s, INFINITY);
        p.f_se2 = (float)(0.25 * P.ea[0] * P.ea[0]);
        // pairs closer than fx_sf: t below it (none where that is below the first
        // edge: they are out of range)
        p.f_sf2 = (float)(P.fx_sf * P.fx_sf);
        double tsf = P.fx_sf * (1.0 + 1e-6);
        if (P.fix == PATH_FIXLOG) tsf = tsf > P.ea[0] ? 2.0 * log2(tsf) * P.fx_inv : -1e3;
        else tsf *= P.fx_inv;
        p.f_close = (float)(P.fx_c + tsf + 0.01);
        if (off && p.f_close < 129.0f) p.f_close = 0.0f;
        for (int a = 0; a < 3; ++a) p.L32[a] = (float)g.L[a];
    }
    // Box tests run in FP32 on coordinates relative to the grids' origins, at
    // most X in magnitude (images included): outward-rounded boxes, and a gap
    // that takes four more roundings of at most 2^-24 x 3 X, so a computed gap
    // exceeds the true one by less than 2^-20 X (2^-50 of the absolute
    // coordinates for the subtraction of the origin); squares and sums add a
    // relative 2^-22.  The limits carry twice that, and seven of the smallest
    // numbers for squares that underflow; they are infinite where a square in reach
    // may overflow, and the tests then drop nothing (catalogues in metres: the FP64
    // kernel counts those as it does any).
    double X = 0.0, A = 0.0, c = 0.0;
    for (int a = 0; a < 3; ++a) {
        X = std::max(X, (hi[a] - lo[a]) + g.L[a]);
        A = std::max({A, fabs(lo[a]), fabs(hi[a])});
        c = std::max(c, g.c[a]);
    }
    const double m = ldexp(X, -19) + ldexp(A, -49);
    p.f_gm = nextafterf((float)m, INFINITY);
    auto up = [&](double r) {
        const double v = (r + m) * (r + m) * (1.0 + ldexp(1.0, -20)) + 1e-44;
        return v < 1e38 ? nextafterf((float)v, INFINITY) : INFINITY;
    };
    p.r2prune = up(P.rcut);
    p.q2prune = p.zprune = INFINITY;
    if (P.mode == PC_BIN_SIGPI) {   // along z: sigma and pi each stay below their last edge
        const double slack = P.rcut - P.reff;
        p.q2prune = up(P.ea[P.na] + slack);
        p.zprune = nextafterf((float)((P.eb[P.nb] + slack + m) * (1.0 + ldexp(1.0, -20)) + 1e-44), INFINITY);
    }
    // absent points: beyond the reach of every point of a neighbouring cell
    // (node), whose offset is at most rcut + 3 c, and small enough for exact floors
    p.far = (float)(4.0 * (P.rcut + c));
}

// Shared-memory layout and launch shape: histogram copies (fewer until they
// fit, else the global histogram), warps per CTA for the most resident warps
// (ties: the smallest CTA).  wint: try the integer weight products first.
static pc_status fit_params(int prec, int opt_priv, int dev, bool weighted, bool wint_try, bool wcorr,
                            PairParams &p, size_t &smem, int &per_sm) {
    int smem_optin = 0;
    PC_CUDA(cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const int static_smem = 256;
    const int lut_size = p.lut_total, path0 = p.path, hs0 = p.hs, nent0 = p.nent;
    const bool f64 = prec == PC_PREC_F64;
    p.f64 = f64 ? 1 : 0;
    p.sm_guess = p.f64;
    const int nw_min = f64 ? 1 : 4;   // as few as still count: edges fill the rest
    auto fit = [&](bool wint) {
        p.wint = wint ? 1 : 0;
        p.wcorr = (wint && wcorr) ? 1 : 0;
        p.path = path0;
        p.layout = LAY_ROWS;
        p.row0 = 0;
        choose_replication(opt_priv, p.nbins, weighted && !wint, p.hist_k);
        if (p.fix && (wint || !weighted)) {   // fixed-point floors (not for binary64 weight sums)
            p.path = p.fix;
            p.row0 = p.fix == PATH_FIX ? 0 : 1;
            if (p.mode == PC_BIN_S) {
                p.layout = LAY_BYTES;
                p.hist_k = 32;
            } else if (!weighted) {
                p.layout = LAY_SKEW;
                p.hist_k = 1;
            } else {   // mu = 1 (pi past its last bin) needs a column of its own
                p.hs = p.n_b + 1;
                p.nent = (p.n_a + p.row0) * p.hs + 1 + p.n_b;
                while (p.hs * p.hist_k > 255) p.hist_k /= 2;   // one byte (f_coef)
            }
        }
        for (;;) {
            p.smem_hist_ok = 1;
            // the floor bins need no tables
            p.lut_total = (p.path != PATH_LUT || f64) ? 0 : lut_size;
            if (pairs_smem(p, nw_min) + static_smem <= (size_t)smem_optin) break;
            if (p.layout == LAY_ROWS && p.hist_k > 1) {   // fewer lane copies, then the global histogram
                p.hist_k /= 2;
                continue;
            }
            p.smem_hist_ok = 0;
            p.path = PATH_LUT;
            p.layout = LAY_ROWS;
            p.row0 = 0;
            p.lut_total = f64 ? 0 : lut_size;
            p.hist_k = 1;
            // many edges: no FP32 roundings beside them
            if (f64 && pairs_smem(p, nw_min) + static_smem > (size_t)smem_optin) p.sm_guess = 0;
            break;
        }
    };
    fit(wint_try && opt_priv != 1);
    if (p.wint && !p.smem_hist_ok) {
        p.hs = hs0;
        p.nent = nent0;
        fit(false);
    }
    {   // the floor paths' pair constants
        auto two = [](float v) { return make_float2(v, v); };
        const float row = 4.0f * p.hist_k * p.hs, col = 4.0f * p.hist_k;
        p.f_coef = (unsigned)p.hist_k | (unsigned)(p.hs * p.hist_k) << 8;
        p.c_23 = two(8388608.0f);
        p.c_p = two(8388607.5f);
        p.c_m1 = two(-1.0f);
        p.c_invA = two(p.path >= PATH_FIX ? p.f_inv : p.lin_invA);
        p.c_offA = two(p.lin_offA);
        p.c_thrA = two(p.lin_thrA);
        p.c_nmS = two(-p.lin_mS);
        p.c_invB = two(p.path >= PATH_FIX ? p.f_invB : (p.mode == PC_BIN_SIGPI ? p.lin_invB2 : p.lin_nB));
        p.c_nmB = two(-p.lin_mA);
        p.c_cB = two(p.mode == PC_BIN_SIGPI ? p.lin_thrB : p.lin_cB);
        p.c_nrow = two(-row);
        p.c_ncol = two(-col);
        p.c_kA = 8388608.0f - (p.path == PATH_LIN ? 0.5f : 1.5f) * row -
                 (p.mode == PC_BIN_S ? 0.0f : 0.5f * col);
    }
    // 8 warps at most with weights: a copy's products between a warp's flushes
    // must hold one batch (64 x 64 products to one lane copy, of WINT_LIMIT 3 / 4 / 8; on
    // one axis 8 a quad and copy, 32 quads, of 4095 / 2 / 8)
    int best_warps = 0, best_nw = 0;
    for (int nw : {1, 2, 4, 8, 12, 16}) {
        if (nw < nw_min || (p.wint && nw > 8)) continue;
        const size_t need = pairs_smem(p, nw);
        if (need + static_smem > (size_t)smem_optin) break;
        const int n = f64 ? pairs_f64_ctas_per_sm(p, need) : pairs_f32_ctas_per_sm(p, need);
        if (n * nw > best_warps) {
            best_warps = n * nw;
            best_nw = nw;
        }
    }
    if (best_nw == 0) {
        if (pairs_smem(p, nw_min) + static_smem > (size_t)smem_optin)
            return fail(PC_EUNSUPPORTED, "bins: tables do not fit in shared memory");
        per_sm = 0;
        return PC_OK;
    }
    smem = pairs_smem(p, best_nw);
    per_sm = best_warps / best_nw;
    return PC_OK;
}

// Kernel parameters and launch shape.
static pc_status make_params(const CountJob &J, const CountSetup &S, const DevBufs &B,
                             PairParams &p, int &grid, size_t &smem) {
    const Plan &P = S.P;
    memset(static_cast<void *>(&p), 0, sizeof(p));
    p.tree = J.tree ? 1 : 0;
    p.tasks = B.tasks;
    p.blocks = B.blocks;
    p.nblocks = B.sc + 1;
    p.work_counter = B.sc;
    p.g = J.geom;
    p.stencil = B.stencil;
    p.nrows = (int)P.stencil.size();
    p.mode = P.mode;
    p.los = P.los;
    p.weighted = S.weighted ? 1 : 0;
    p.n_a = P.na;
    p.n_b = P.nb;
    p.nbins = P.nbins;
    p.r2cut = P.r2cut;
    p.lut = B.lut;
    p.lut_total = (int)P.lut.size();
    p.la = P.la;
    p.lb = P.lb;
    p.eps_a = P.eps_a;
    p.eps_b = P.eps_b;
    p.mu_A = P.mu_A;
    p.mu_B = P.mu_B;
    p.mu_W = P.mu_W;
    p.Ea = B.ea;
    p.Eb = B.eb;
    p.hist = B.hist;
    p.whist = B.whist;
    p.queue = B.queue;
    p.qcount = B.ctr + 2;
    p.qcap = S.qcap;
    p.counters = B.ctr;
    p.shard_count = S.o.shard_count > 1 ? S.o.shard_count : 1;
    p.shard_index = S.o.shard_count > 1 ? S.o.shard_index : 0;
    set_fp32_params(J.geom, J.lo, J.hi, P, S.prec, p);
    p.nsub = (S.bi + 63) / 64;
    p.multi = J.nhist > 1 ? 1 : 0;
    for (auto &t : J.tasks) p.npts_i += t.gi.n;
    p.npts_i /= p.shard_count;
    // integer weight products need floor bins, every weight packable and
    // shared histograms
    const bool wint_try = S.weighted && (p.path != PATH_LUT || p.fix) && J.wint_ok && S.prec == PC_PREC_F32_RESCUE;
    int per_sm = 0;
    pc_status s = fit_params(S.prec, S.o.priv, S.dev, S.weighted, wint_try, J.wcorr, p, smem, per_sm);
    if (s != PC_OK) return s;
    int dev_sms = 0;
    PC_CUDA(cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, S.dev));
    if (per_sm <= 0)
        return fail(PC_ECUDA, std::string("pair kernel cannot be resident: ") + pc_last_error());
    if (S.o.grid_ctas_per_sm > 0) per_sm = std::min(per_sm, S.o.grid_ctas_per_sm);
    grid = dev_sms * per_sm;
    return PC_OK;
}

// Device work of one count, in stream order (also what a captured graph
// replays): clear, block list, pair kernel, rescue kernel.
static pc_status enqueue_count(const CountSetup &S, const DevBufs &B, const PairParams &p, int grid,
                               size_t smem, cudaStream_t st, cudaEvent_t ev_pairs,
                               cudaEvent_t ev_rescue, cudaEvent_t ev_done,
                               const std::function<cudaError_t()> &tree_blocks_fn = {}) {
    PC_CUDA(cudaMemsetAsync(B.hist, 0, sizeof(unsigned long long) * S.hist_n, st));
    if (S.weighted) PC_CUDA(cudaMemsetAsync(B.whist, 0, sizeof(double) * S.hist_n, st));
    PC_CUDA(cudaMemsetAsync(B.ctr, 0, sizeof(unsigned long long) * 4, st));
    PC_CUDA(cudaMemsetAsync(B.sc, 0, sizeof(int) * 4, st));
    if (tree_blocks_fn)   // tree counts: balanced blocks of the list nodes
        PC_CUDA(tree_blocks_fn());
    else
        PC_CUDA(make_blocks_into(B.tasks, S.ntasks, S.ncell, S.bi, p.shard_index, p.shard_count,
                                 B.blocks, B.sc + 1, B.cnt,
                                 B.off, B.tot, st));
    if (ev_pairs) PC_CUDA(cudaEventRecord(ev_pairs, st));
    cudaError_t e = (S.prec == PC_PREC_F64) ? launch_pairs_f64(p, grid, smem, st)
                                            : launch_pairs_f32(p, grid, smem, st);
    if (e != cudaSuccess) return cuda_fail(e, "pair kernel launch");
    if (ev_rescue) PC_CUDA(cudaEventRecord(ev_rescue, st));
    if (S.prec == PC_PREC_F32_RESCUE && S.qcap) {
        e = launch_rescue(p, st);
        if (e != cudaSuccess) return cuda_fail(e, "rescue kernel launch");
    }
    if (ev_done) PC_CUDA(cudaEventRecord(ev_done, st));
    return PC_OK;
}

static void copy_out(void *dst, const void *src, size_t bytes, cudaStream_t st, cudaError_t &e) {
    if (!dst || e != cudaSuccess) return;
    cudaMemcpyKind k = is_device_ptr(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    e = cudaMemcpyAsync(dst, src, bytes, k, st);
}

static void fill_stats(pc_stats *stats, const CountSetup &S, double cell_size,
                       const unsigned long long hc[4], int hblk, float ms_total, float ms_pairs,
                       float ms_rescue, long long launches) {
    if (!stats) return;
    memset(stats, 0, sizeof(*stats));
    stats->candidates = (long long)hc[0];
    stats->rescue_inline = (long long)hc[1];
    stats->pruned = (long long)hc[3];
    stats->prec = S.prec;
    stats->wsum = S.wsum;
    stats->rescued = (long long)std::min<unsigned long long>(hc[2], S.qcap) + (long long)hc[1];
    stats->blocks = hblk;
    stats->cell_size = cell_size;
    stats->ms_total = ms_total;
    stats->ms_pairs = ms_pairs;
    stats->ms_rescue = ms_rescue;
    stats->launches = (int)launches;
}

struct Events {
    cudaEvent_t e[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    bool on = false;
    explicit Events(bool want) : on(want) {
        if (on) for (auto &x : e) cudaEventCreate(&x);
    }
    ~Events() {
        if (on) for (auto &x : e) cudaEventDestroy(x);
    }
    float ms(int a, int b) const {
        float m = 0.f;
        if (on) cudaEventElapsedTime(&m, e[a], e[b]);
        return m;
    }
};

static pc_status run_count(const CountJob &J, const pc_bins *b, const pc_opts *opt,
                           cudaStream_t st, long long *counts, double *wcounts, pc_stats *stats) {
    CountSetup S;
    pc_status s = setup_count(J, b, opt, wcounts != nullptr, S);
    if (s != PC_OK) return s;
    DevBufs B;
    s = ensure_bufs(workspace(S.dev), S, B);
    if (s != PC_OK) return s;
    PairParams p;
    int grid = 0;
    size_t smem = 0;
    s = make_params(J, S, B, p, grid, smem);
    if (s == PC_OK) s = attach_wsums(workspace(S.dev), p, grid);
    if (s != PC_OK) return s;
    S.wsum = p.wint ? (p.wcorr ? 3 : 2) : (S.weighted ? 1 : 0);
    Events ev(stats != nullptr);
    const long long launches0 = launch_count();
    if (ev.on) PC_CUDA(cudaEventRecord(ev.e[0], st));
    s = upload_tables(J, S, B, st);
    if (s != PC_OK) return s;
    s = enqueue_count(S, B, p, grid, smem, st, ev.e[1], ev.e[2], ev.e[3]);
    if (s != PC_OK) return s;
    cudaError_t e = cudaSuccess;
    copy_out(counts, B.hist, sizeof(long long) * S.hist_n, st, e);
    copy_out(wcounts, B.whist, sizeof(double) * S.hist_n, st, e);
    if (e != cudaSuccess) return cuda_fail(e, "result copy");
    unsigned long long hc[4] = {0, 0, 0, 0};
    int hblk = 0;
    if (ev.on) {
        PC_CUDA(cudaMemcpyAsync(hc, B.ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
        PC_CUDA(cudaMemcpyAsync(&hblk, B.sc + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        PC_CUDA(cudaEventRecord(ev.e[4], st));
    }
    PC_CUDA(cudaStreamSynchronize(st));
    fill_stats(stats, S, J.cell_size, hc, hblk, ev.ms(0, 4), ev.ms(1, 2), ev.ms(2, 3),
               launch_count() - launches0);
    return PC_OK;
}

// ---------------------------------------------------------------------------
// captured count graphs (pc_count_batch with use_graph)
// ---------------------------------------------------------------------------
// A graph owns its buffers: the shared workspace may be reallocated by other
// calls, and a graph must keep the addresses it was captured with.
struct GraphEntry {
    int dev = 0;
    std::vector<const pc_grid *> grids;
    int mode = 0, los = 0;
    std::vector<double> ea, eb;
    pc_opts o;
    bool weighted = false;
    Workspace W;
    CountSetup S;
    DevBufs B;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    unsigned long long *h_hist = nullptr;   // pinned copies written by the graph
    double *h_whist = nullptr;
    unsigned long long *h_ctr = nullptr;
    int *h_blocks = nullptr;
    long long kernels = 0;                  // kernel launches inside the graph
    ~GraphEntry() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        cudaFreeHost(h_hist);
        cudaFreeHost(h_whist);
        cudaFreeHost(h_ctr);
        cudaFreeHost(h_blocks);
        for (Buf *b : {&W.hist, &W.whist, &W.counters, &W.scalars, &W.queue, &W.blocks, &W.tmp_cnt,
                       &W.tmp_off, &W.tmp_tot, &W.tasks, &W.stencil, &W.lut, &W.ea, &W.eb, &W.wsums})
            if (b->p) cudaFree(b->p);
    }
};

static std::vector<std::unique_ptr<GraphEntry>> &graph_cache() {
    static std::vector<std::unique_ptr<GraphEntry>> c;
    return c;
}

// Drop every cached graph that uses grid g (called when g is freed).
void forget_grid(const pc_grid *g) {
    auto &c = graph_cache();
    for (size_t k = 0; k < c.size();) {
        bool uses = false;
        for (auto *x : c[k]->grids) uses = uses || (x == g);
        if (uses) c.erase(c.begin() + k); else ++k;
    }
}

static bool same_opts(const pc_opts &a, const pc_opts &b) {
    return a.prec == b.prec && a.cell_size == b.cell_size && a.ipt == b.ipt && a.priv == b.priv &&
           a.rescue_capacity == b.rescue_capacity && a.grid_ctas_per_sm == b.grid_ctas_per_sm &&
           a.shard_index == b.shard_index && a.shard_count == b.shard_count;
}

static pc_status run_count_graph(const CountJob &J, const std::vector<const pc_grid *> &grids,
                                 const pc_bins *b, const pc_opts *opt, cudaStream_t st,
                                 long long *counts, double *wcounts, pc_stats *stats) {
    pc_opts o;
    memset(&o, 0, sizeof(o));
    o.priv = -1;
    if (opt) o = *opt;
    const bool weighted = wcounts != nullptr;
    if (!b || !b->edges_a || (b->mode != PC_BIN_S && !b->edges_b))
        return fail(PC_EINVAL, "bins: missing edges");
    std::vector<double> ea(b->edges_a, b->edges_a + std::max(b->n_a, 0) + 1);
    std::vector<double> eb;
    if (b->mode != PC_BIN_S) eb.assign(b->edges_b, b->edges_b + std::max(b->n_b, 0) + 1);
    GraphEntry *G = nullptr;
    for (auto &c : graph_cache())
        if (c->dev == J.device && c->grids == grids && c->mode == b->mode && c->los == b->los &&
            c->ea == ea && c->eb == eb && same_opts(c->o, o) && c->weighted == weighted)
            G = c.get();
    const long long launches0 = launch_count();
    if (!G) {
        std::unique_ptr<GraphEntry> N(new GraphEntry());
        N->dev = J.device;
        N->grids = grids;
        N->mode = b->mode;
        N->los = b->los;
        N->ea = ea;
        N->eb = eb;
        N->o = o;
        N->weighted = weighted;
        pc_status s = setup_count(J, b, &o, weighted, N->S);
        if (s != PC_OK) return s;
        s = ensure_bufs(N->W, N->S, N->B);
        if (s != PC_OK) return s;
        PairParams p;
        int grid = 0;
        size_t smem = 0;
        s = make_params(J, N->S, N->B, p, grid, smem);
        if (s == PC_OK) s = attach_wsums(N->W, p, grid);
        if (s != PC_OK) return s;
        N->S.wsum = p.wint ? (p.wcorr ? 3 : 2) : (N->S.weighted ? 1 : 0);
        const size_t hb = N->S.hist_n;
        PC_CUDA(::pc::alloc_host(&N->h_hist, sizeof(unsigned long long) * hb));
        if (weighted) PC_CUDA(::pc::alloc_host(&N->h_whist, sizeof(double) * hb));
        PC_CUDA(::pc::alloc_host(&N->h_ctr, sizeof(unsigned long long) * 4));
        PC_CUDA(::pc::alloc_host(&N->h_blocks, sizeof(int)));
        cudaStream_t cap = nullptr;
        PC_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        s = upload_tables(J, N->S, N->B, cap);
        if (s == PC_OK) {
            cudaError_t e = cudaStreamSynchronize(cap);
            if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
            if (e != cudaSuccess) s = cuda_fail(e, "graph capture");
        }
        if (s == PC_OK) {
            const long long k0 = launch_count();
            s = enqueue_count(N->S, N->B, p, grid, smem, cap, nullptr, nullptr, nullptr);
            N->kernels = launch_count() - k0;
            cudaError_t e = cudaSuccess;
            if (s == PC_OK) {
                e = cudaMemcpyAsync(N->h_hist, N->B.hist, sizeof(unsigned long long) * hb,
                                    cudaMemcpyDeviceToHost, cap);
                if (e == cudaSuccess && weighted)
                    e = cudaMemcpyAsync(N->h_whist, N->B.whist, sizeof(double) * hb,
                                        cudaMemcpyDeviceToHost, cap);
                if (e == cudaSuccess)
                    e = cudaMemcpyAsync(N->h_ctr, N->B.ctr, sizeof(unsigned long long) * 4,
                                        cudaMemcpyDeviceToHost, cap);
                if (e == cudaSuccess)
                    e = cudaMemcpyAsync(N->h_blocks, N->B.sc + 1, sizeof(int),
                                        cudaMemcpyDeviceToHost, cap);
            }
            cudaError_t e2 = cudaStreamEndCapture(cap, &N->graph);
            if (s == PC_OK && e != cudaSuccess) s = cuda_fail(e, "graph capture copy");
            if (s == PC_OK && e2 != cudaSuccess) s = cuda_fail(e2, "graph capture end");
            if (s == PC_OK) {
                e = cudaGraphInstantiate(&N->exec, N->graph, 0);
                if (e != cudaSuccess) s = cuda_fail(e, "graph instantiate");
            }
        }
        cudaStreamDestroy(cap);
        if (s != PC_OK) return s;
        graph_cache().push_back(std::move(N));
        G = graph_cache().back().get();
    }
    Events ev(stats != nullptr);
    if (ev.on) PC_CUDA(cudaEventRecord(ev.e[0], st));
    PC_CUDA(cudaGraphLaunch(G->exec, st));
    note_launch((int)G->kernels);   // a replay launches the captured kernels again
    if (ev.on) PC_CUDA(cudaEventRecord(ev.e[4], st));
    PC_CUDA(cudaStreamSynchronize(st));
    const size_t hb = G->S.hist_n;
    cudaError_t e = cudaSuccess;
    if (counts) {
        if (is_device_ptr(counts))
            e = cudaMemcpy(counts, G->h_hist, sizeof(long long) * hb, cudaMemcpyHostToDevice);
        else
            memcpy(counts, G->h_hist, sizeof(long long) * hb);
    }
    if (wcounts && e == cudaSuccess) {
        if (is_device_ptr(wcounts))
            e = cudaMemcpy(wcounts, G->h_whist, sizeof(double) * hb, cudaMemcpyHostToDevice);
        else
            memcpy(wcounts, G->h_whist, sizeof(double) * hb);
    }
    if (e != cudaSuccess) return cuda_fail(e, "result copy");
    unsigned long long hc[4] = {G->h_ctr[0], G->h_ctr[1], G->h_ctr[2], G->h_ctr[3]};
    fill_stats(stats, G->S, J.cell_size, hc, *G->h_blocks, ev.ms(0, 4), 0.f, 0.f,
               launch_count() - launches0);
    return PC_OK;
}

static TaskDev task_of(const pc_grid *gi, const pc_grid *gj, int hist, int is_auto) {
    TaskDev t;
    t.gi = GridDev{gi->rel, gi->cx, gi->xw, gi->cell_start, gi->n, gi->wlo, gi->obox,
                   {gi->g.lo[0], gi->g.lo[1], gi->g.lo[2]}};
    t.gj = GridDev{gj->rel, gj->cx, gj->xw, gj->cell_start, gj->n, gj->wlo, gj->obox,
                   {gj->g.lo[0], gj->g.lo[1], gj->g.lo[2]}};
    t.hist = hist;
    t.is_auto = is_auto;
    // one unit of the integer weight products: 2^(emax_i + emax_j - 300)
    // (w = M 2^(e - 150) with the 24-bit significand M and biased exponent e);
    // the packed significands' product is shifted down by both ranges
    t.wscale = (gi->wint && gj->wint) ? ldexp(1.0, gi->wemax + gj->wemax - 300) : 0.0;
    return t;
}

static bool same_geometry(const pc_grid *a, const pc_grid *b) {
    if (a->g.periodic != b->g.periodic) return false;
    for (int k = 0; k < 3; ++k) {
        if (a->g.ng[k] != b->g.ng[k] || a->g.c[k] != b->g.c[k] || a->g.lo[k] != b->g.lo[k] ||
            a->g.L[k] != b->g.L[k])
            return false;
    }
    return a->device == b->device;
}

}  // namespace pc

using namespace pc;

extern "C" pc_status pc_count_auto(const pc_grid *g, const pc_bins *b, const pc_opts *o,
                                   void *stream, long long *counts, double *wcounts,
                                   pc_stats *st) {
    std::lock_guard<std::mutex> lk(api_mutex());
    if (!g) return fail(PC_EINVAL, "pc_count_auto: grid is NULL");
    if (!counts && !wcounts) return fail(PC_EINVAL, "pc_count_auto: no output buffer");
    if (wcounts && !g->weighted) return fail(PC_EINVAL, "pc_count_auto: grid has no weights");
    CountJob J;
    J.tasks.push_back(task_of(g, g, 0, 1));
    J.nhist = 1;
    J.is_auto = true;
    job_set_grid(J, g);
    job_add_bounds(J, g, true);
    job_add_wint(J, g, g);
    return run_count(J, b, o, (cudaStream_t)stream, counts, wcounts, st);
}

extern "C" pc_status pc_count_cross(const pc_grid *g1, const pc_grid *g2, const pc_bins *b,
                                    const pc_opts *o, void *stream, long long *counts,
                                    double *wcounts, pc_stats *st) {
    std::lock_guard<std::mutex> lk(api_mutex());
    if (!g1 || !g2) return fail(PC_EINVAL, "pc_count_cross: grid is NULL");
    if (!counts && !wcounts) return fail(PC_EINVAL, "pc_count_cross: no output buffer");
    if (!same_geometry(g1, g2))
        return fail(PC_EINVAL, "pc_count_cross: grids differ in box, bounds or cell size");
    if (wcounts && !(g1->weighted && g2->weighted))
        return fail(PC_EINVAL, "pc_count_cross: both grids need weights for weighted counts");
    // Every pair is symmetric.  The denser catalogue gives the i-points: its 64 points
    // fill a warp and span a small box, so fewer boxes of the other come within reach.
    // But where the other has fewer than two points a cell, its runs of eight are
    // mostly points of other rows, and it gives them (10^6 points and n, pairs up to
    // 150 in cells of 60, the pair kernel: n = 1,000 0.36 -> 0.18 ms, 4,000 (one a cell)
    // 0.61 -> 0.47, 16,000 1.08 against 1.37; to 40 in cells of 20: 150,000 (1.2) 2.4 ->
    // 1.3).  Shards are cells of g1, so they keep it
    if (!(o && o->shard_count > 1)) {
        const bool sparse = std::min(g1->n, g2->n) < 2ll * g1->ncell;
        if (sparse ? g2->n < g1->n : g2->n > g1->n) std::swap(g1, g2);
    }
    CountJob J;
    J.tasks.push_back(task_of(g1, g2, 0, 0));
    J.nhist = 1;
    J.is_auto = false;
    job_set_grid(J, g1);
    job_add_bounds(J, g1, true);
    job_add_bounds(J, g2, false);
    job_add_wint(J, g1, g2);
    return run_count(J, b, o, (cudaStream_t)stream, counts, wcounts, st);
}

extern "C" pc_status pc_count_batch(const pc_grid *const *gs, int m, const pc_bins *b,
                                    const pc_opts *o, void *stream, long long *counts,
                                    double *wcounts, pc_stats *st) {
    std::lock_guard<std::mutex> lk(api_mutex());
    if (!gs || m <= 0) return fail(PC_EINVAL, "pc_count_batch: no grids");
    if (m >= (1 << 26)) return fail(PC_EOVERFLOW, "pc_count_batch: too many grids");
    if (!counts && !wcounts) return fail(PC_EINVAL, "pc_count_batch: no output buffer");
    CountJob J;
    for (int k = 0; k < m; ++k) {
        if (!gs[k]) return fail(PC_EINVAL, "pc_count_batch: grid is NULL");
        if (!same_geometry(gs[0], gs[k]))
            return fail(PC_EINVAL, "pc_count_batch: grids differ in box or cell size");
        if (wcounts && !gs[k]->weighted) return fail(PC_EINVAL, "pc_count_batch: grid has no weights");
        J.tasks.push_back(task_of(gs[k], gs[k], k, 1));
        job_add_bounds(J, gs[k], k == 0);
        job_add_wint(J, gs[k], gs[k]);
    }
    J.nhist = m;
    J.is_auto = true;
    job_set_grid(J, gs[0]);
    if (o && o->use_graph) {
        std::vector<const pc_grid *> grids(gs, gs + m);
        return run_count_graph(J, grids, b, o, (cudaStream_t)stream, counts, wcounts, st);
    }
    return run_count(J, b, o, (cudaStream_t)stream, counts, wcounts, st);
}

// ---------------------------------------------------------------------------
// k-d tree counts (Alg. 3): the traversal lists the block pairs, then the
// same pair and rescue kernels as the grid path run over them
// ---------------------------------------------------------------------------
static bool same_tree_geometry(const pc_tree *a, const pc_tree *b) {
    if (a->g.periodic != b->g.periodic || a->device != b->device) return false;
    for (int k = 0; k < 3; ++k)
        if (a->g.L[k] != b->g.L[k]) return false;
    return true;
}

static GridDev tree_dev(const pc_tree *t) {
    return GridDev{t->rel, nullptr, t->xw, nullptr, t->n, t->wlo, t->obox,
                   {t->g.lo[0], t->g.lo[1], t->g.lo[2]}};
}

static double tree_rmin(const pc_tree *t) {
    if (t->g.periodic || !(t->r2min > 0.0)) return 0.0;
    return sqrt(t->r2min) * (1.0 - 1e-12);
}

extern "C" pc_status pc_count_tree(const pc_tree *t1, const pc_tree *t2, const pc_bins *b,
                                   const pc_opts *opt, void *stream, long long *counts,
                                   double *wcounts, pc_stats *stats) {
    std::lock_guard<std::mutex> lk(api_mutex());
    if (!t1) return fail(PC_EINVAL, "pc_count_tree: tree is NULL");
    if (!counts && !wcounts) return fail(PC_EINVAL, "pc_count_tree: no output buffer");
    const bool is_auto = (t2 == nullptr);
    const pc_tree *tj = is_auto ? t1 : t2;
    if (!same_tree_geometry(t1, tj))
        return fail(PC_EINVAL, "pc_count_tree: trees differ in box or device");
    if (wcounts && !(t1->weighted && tj->weighted))
        return fail(PC_EINVAL, "pc_count_tree: weighted counts need weights on every tree");
    cudaStream_t st = (cudaStream_t)stream;
    // the denser catalogue gives the i-points (see pc_count_cross)
    if (!is_auto && !(opt && opt->shard_count > 1) && tj->n > t1->n) std::swap(t1, tj);

    CountJob J;
    TaskDev T;
    T.gi = tree_dev(t1);
    T.gj = tree_dev(tj);
    T.hist = 0;
    T.is_auto = is_auto ? 1 : 0;
    T.wscale = (t1->wint && tj->wint) ? ldexp(1.0, t1->wemax + tj->wemax - 300) : 0.0;
    J.tasks.push_back(T);
    J.nhist = 1;
    J.is_auto = is_auto;
    J.tree = true;
    // the error bands take the largest block extent where the grid takes
    // the cell side (point offsets from their block centre are at most half
    // of it)
    J.geom = t1->g;
    const double cb = std::max(t1->bext, tj->bext);
    for (int a = 0; a < 3; ++a) {
        J.geom.c[a] = std::max(cb, 1e-300);
        J.geom.c32[a] = (float)J.geom.c[a];
        J.lo[a] = std::min(t1->pts_lo[a], tj->pts_lo[a]);
        J.hi[a] = std::max(t1->pts_hi[a], tj->pts_hi[a]);
        J.plo[a] = J.lo[a];
        J.phi[a] = J.hi[a];
    }
    J.rmin = std::min(tree_rmin(t1), tree_rmin(tj));
    J.device = t1->device;
    J.cell_size = cb;
    if (!t1->wint || !tj->wint ||
        (t1->wemax - t1->wemin) + (tj->wemax - tj->wemin) > WINT_MAX_SPAN)
        J.wint_ok = false;
    if (t1->wcorr || tj->wcorr) J.wcorr = true;

    pc_opts o;
    memset(&o, 0, sizeof(o));
    o.priv = -1;
    if (opt) o = *opt;
    o.ipt = (o.ipt == 4) ? 4 : 2;
    J.ncell = (1 << t1->blevel) * tree_chunks(t1, o.ipt);   // i-blocks (buffer sizes)
    CountSetup S;
    pc_status s = setup_count(J, b, &o, wcounts != nullptr, S);
    if (s != PC_OK) return s;
    if (S.prec != PC_PREC_F32_RESCUE)
        return fail(PC_EUNSUPPORTED,
                    "pc_count_tree: runs the FP32 + rescue kernel only (the plain FP64 path, "
                    "asked for or forced by a midpoint line of sight close to the observer or a reach "
                    "above 1.7e19, "
                    "is a grid-path option)");
    DevBufs B;
    s = ensure_bufs(workspace(S.dev), S, B);
    if (s != PC_OK) return s;
    PairParams p;
    int grid = 0;
    size_t smem = 0;
    s = make_params(J, S, B, p, grid, smem);
    if (s == PC_OK) s = attach_wsums(workspace(S.dev), p, grid);
    if (s != PC_OK) return s;
    S.wsum = p.wint ? (p.wcorr ? 3 : 2) : (S.weighted ? 1 : 0);
    Events ev(stats != nullptr);
    const long long launches0 = launch_count();
    if (ev.on) PC_CUDA(cudaEventRecord(ev.e[0], st));
    // node pairs closer than the candidate cut, farther than the smallest
    // s edge (the box bounds are exact up to rounding: relative margins)
    const double r2hi = (double)S.P.r2cut * (1.0 + 1e-9);
    const double r2lo = (S.P.mode != PC_BIN_SIGPI) ? S.P.Ea[0] * (1.0 - 1e-9) : 0.0;
    TreeLists TL;
    s = tree_traverse(t1, tj, is_auto, r2hi, r2lo, st, TL);
    if (s != PC_OK) return s;
    p.tseg = TL.seg;
    p.tseg_off = TL.seg_off;
    p.tblk_j = tj->brng;
    p.tcen_i = t1->bcen;
    p.tcen_j = tj->bcen;
    s = upload_tables(J, S, B, st);
    if (s != PC_OK) return s;
    s = enqueue_count(S, B, p, grid, smem, st, ev.e[1], ev.e[2], ev.e[3],
                      [&]() {
                          return tree_blocks(t1, S.ipt, p.shard_index, p.shard_count, B.blocks,
                                             B.sc + 1, st);
                      });
    if (s != PC_OK) return s;
    cudaError_t e = cudaSuccess;
    copy_out(counts, B.hist, sizeof(long long) * S.hist_n, st, e);
    copy_out(wcounts, B.whist, sizeof(double) * S.hist_n, st, e);
    if (e != cudaSuccess) return cuda_fail(e, "result copy");
    unsigned long long hc[4] = {0, 0, 0, 0};
    int hblk = 0;
    if (ev.on) {
        PC_CUDA(cudaMemcpyAsync(hc, B.ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
        PC_CUDA(cudaMemcpyAsync(&hblk, B.sc + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        PC_CUDA(cudaEventRecord(ev.e[4], st));
    }
    PC_CUDA(cudaStreamSynchronize(st));
    fill_stats(stats, S, J.cell_size, hc, hblk, ev.ms(0, 4), ev.ms(1, 2), ev.ms(2, 3),
               launch_count() - launches0);
    if (stats) {
        stats->tree_pairs = TL.npairs;
        stats->ms_traverse = ev.ms(0, 1);
    }
    return PC_OK;
}

// Auto counts of m trees in one pair-kernel launch (the tree path's batch):
// each tree is traversed on its own and its lists appended to the batch's.
extern "C" pc_status pc_count_tree_batch(const pc_tree *const *ts, int m, const pc_bins *b,
                                         const pc_opts *opt, void *stream, long long *counts,
                                         double *wcounts, pc_stats *stats) {
    std::lock_guard<std::mutex> lk(api_mutex());
    if (!ts || m <= 0) return fail(PC_EINVAL, "pc_count_tree_batch: no trees");
    if (m >= (1 << 26)) return fail(PC_EOVERFLOW, "pc_count_tree_batch: too many trees");
    if (!counts && !wcounts) return fail(PC_EINVAL, "pc_count_tree_batch: no output buffer");
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<const pc_tree *> trees(ts, ts + m);
    CountJob J;
    double cb = 0.0;
    J.wint_ok = true;
    long long nlist = 0;
    pc_opts o;
    memset(&o, 0, sizeof(o));
    o.priv = -1;
    if (opt) o = *opt;
    o.ipt = (o.ipt == 4) ? 4 : 2;
    for (int k = 0; k < m; ++k) {
        const pc_tree *t = trees[k];
        if (!t) return fail(PC_EINVAL, "pc_count_tree_batch: tree is NULL");
        if (!same_tree_geometry(trees[0], t))
            return fail(PC_EINVAL, "pc_count_tree_batch: trees differ in box or device");
        if (wcounts && !t->weighted)
            return fail(PC_EINVAL, "pc_count_tree_batch: weighted counts need weights on every tree");
        TaskDev T;
        T.gi = tree_dev(t);
        T.gj = T.gi;
        T.hist = k;
        T.is_auto = 1;
        T.wscale = t->wint ? ldexp(1.0, 2 * t->wemax - 300) : 0.0;
        J.tasks.push_back(T);
        cb = std::max(cb, t->bext);
        for (int a = 0; a < 3; ++a) {
            J.lo[a] = k ? std::min(J.lo[a], t->pts_lo[a]) : t->pts_lo[a];
            J.hi[a] = k ? std::max(J.hi[a], t->pts_hi[a]) : t->pts_hi[a];
        }
        J.rmin = k ? std::min(J.rmin, tree_rmin(t)) : tree_rmin(t);
        if (!t->wint || 2 * (t->wemax - t->wemin) > WINT_MAX_SPAN) J.wint_ok = false;
        if (t->wcorr) J.wcorr = true;
        nlist += (long long)(1 << t->blevel) * tree_chunks(t, o.ipt);
    }
    if (nlist >= (1LL << 31)) return fail(PC_EOVERFLOW, "pc_count_tree_batch: too many blocks");
    J.nhist = m;
    J.is_auto = true;
    J.tree = true;
    J.geom = trees[0]->g;
    for (int a = 0; a < 3; ++a) {
        J.geom.c[a] = std::max(cb, 1e-300);
        J.geom.c32[a] = (float)J.geom.c[a];
        J.plo[a] = J.lo[a];
        J.phi[a] = J.hi[a];
    }
    J.device = trees[0]->device;
    // buffers are sized per task x cells: ntasks * ncell covers the blocks
    J.ncell = (int)((nlist + m - 1) / m);
    J.cell_size = cb;
    CountSetup S;
    pc_status s = setup_count(J, b, &o, wcounts != nullptr, S);
    if (s != PC_OK) return s;
    if (S.prec != PC_PREC_F32_RESCUE)
        return fail(PC_EUNSUPPORTED,
                    "pc_count_tree_batch: runs the FP32 + rescue kernel only (see pc_count_tree)");
    DevBufs B;
    s = ensure_bufs(workspace(S.dev), S, B);
    if (s != PC_OK) return s;
    PairParams p;
    int grid = 0;
    size_t smem = 0;
    s = make_params(J, S, B, p, grid, smem);
    if (s == PC_OK) s = attach_wsums(workspace(S.dev), p, grid);
    if (s != PC_OK) return s;
    S.wsum = p.wint ? (p.wcorr ? 3 : 2) : (S.weighted ? 1 : 0);
    Events ev(stats != nullptr);
    const long long launches0 = launch_count();
    if (ev.on) PC_CUDA(cudaEventRecord(ev.e[0], st));
    static std::map<int, TreeBatch> batches;   // per device, reused (calls are serialised)
    TreeBatch &TB = batches[S.dev];
    const double r2hi = (double)S.P.r2cut * (1.0 + 1e-9);
    const double r2lo = (S.P.mode != PC_BIN_SIGPI) ? S.P.Ea[0] * (1.0 - 1e-9) : 0.0;
    s = tree_batch_lists(trees, S.ipt, r2hi, r2lo, st, TB);
    if (s != PC_OK) return s;
    p.tseg = (const int2 *)TB.seg.p;
    p.tseg_off = (const int *)TB.off.p;
    p.tblk_j = (const int2 *)TB.rng.p;
    p.tcen_i = (const double *)TB.cen.p;
    p.tcen_j = (const double *)TB.cen.p;
    s = upload_tables(J, S, B, st);
    if (s != PC_OK) return s;
    s = enqueue_count(S, B, p, grid, smem, st, ev.e[1], ev.e[2], ev.e[3], [&]() {
        return tree_blocks_batch(trees, TB, S.ipt, p.shard_index, p.shard_count, B.blocks,
                                 B.sc + 1, st);
    });
    if (s != PC_OK) return s;
    cudaError_t e = cudaSuccess;
    copy_out(counts, B.hist, sizeof(long long) * S.hist_n, st, e);
    copy_out(wcounts, B.whist, sizeof(double) * S.hist_n, st, e);
    if (e != cudaSuccess) return cuda_fail(e, "result copy");
    unsigned long long hc[4] = {0, 0, 0, 0};
    int hblk = 0;
    if (ev.on) {
        PC_CUDA(cudaMemcpyAsync(hc, B.ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
        PC_CUDA(cudaMemcpyAsync(&hblk, B.sc + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        PC_CUDA(cudaEventRecord(ev.e[4], st));
    }
    PC_CUDA(cudaStreamSynchronize(st));
    fill_stats(stats, S, J.cell_size, hc, hblk, ev.ms(0, 4), ev.ms(1, 2), ev.ms(2, 3),
               launch_count() - launches0);
    if (stats) {
        stats->tree_pairs = TB.npairs;
        stats->ms_traverse = ev.ms(0, 1);
    }
    return PC_OK;
}

// Host-only view of the stencil the grid path enumerates (no device work).
extern "C" pc_status pc_stencil(const double cell[3], double r_max, int half, int max_rows,
                                int *rows, int *n_rows) {
    if (!cell || !n_rows || max_rows < 0 || (max_rows > 0 && !rows))
        return fail(PC_EINVAL, "pc_stencil: bad arguments");
    if (!(r_max > 0.0) || !std::isfinite(r_max))
        return fail(PC_EINVAL, "pc_stencil: r_max must be positive and finite");
    Geom g;
    memset(&g, 0, sizeof(g));
    for (int a = 0; a < 3; ++a) {
        if (!(cell[a] > 0.0) || !std::isfinite(cell[a]))
            return fail(PC_EINVAL, "pc_stencil: cell sides must be positive and finite");
        if (r_max / cell[a] > 4096.0) return fail(PC_EOVERFLOW, "pc_stencil: too many cells per axis");
        g.c[a] = cell[a];
        g.ng[a] = 1;
    }
    std::vector<int4> st;
    int kmax[3];
    build_stencil(g, r_max, half != 0, st, kmax);
    *n_rows = (int)st.size();
    if ((int)st.size() > max_rows) return fail(PC_EOVERFLOW, "pc_stencil: max_rows too small");
    for (size_t k = 0; k < st.size(); ++k) {
        rows[4 * k] = st[k].x;
        rows[4 * k + 1] = st[k].y;
        rows[4 * k + 2] = st[k].z;
        rows[4 * k + 3] = st[k].w;
    }
    return PC_OK;
}

// Host-only view of the FP32 path's error bands and bin decisions for a
// count (no device work): make_plan on a geometry built from the arguments.
extern "C" pc_status pc_fp32_bands(const pc_bins *b, const double cell[3], const double lo[3],
                                   const double hi[3], const double L[3], int periodic,
                                   double rmin, double out[19]) {
    if (!b || !cell || !lo || !hi || !out || (periodic && !L))
        return fail(PC_EINVAL, "pc_fp32_bands: bad arguments");
    Geom g;
    memset(&g, 0, sizeof(g));
    g.periodic = periodic ? 1 : 0;
    for (int a = 0; a < 3; ++a) {
        if (!(cell[a] > 0.0) || !std::isfinite(cell[a]) || !std::isfinite(lo[a]) ||
            !std::isfinite(hi[a]) || hi[a] < lo[a])
            return fail(PC_EINVAL, "pc_fp32_bands: bad cell sides or bounds");
        if (periodic && (!(L[a] > 0.0) || !std::isfinite(L[a])))
            return fail(PC_EINVAL, "pc_fp32_bands: periodic box needs L > 0");
        g.c[a] = cell[a];
        g.c32[a] = (float)cell[a];
        g.ng[a] = 1;
        g.lo[a] = lo[a];
        g.L[a] = periodic ? L[a] : 0.0;
        g.hL[a] = 0.5 * g.L[a];
    }
    Plan P;
    pc_status s = make_plan(b, g, lo, hi, rmin, false, P, false);
    if (s != PC_OK) return s;
    out[0] = P.eps_a;
    out[1] = P.eps_b;
    out[2] = P.mu_A;
    out[3] = P.mu_B;
    out[4] = P.rcut;
    out[5] = P.fp32_ok;
    out[6] = P.lin;
    out[7] = P.r2cut;
    // packed floors (pc_fp32_floors has what a kernel receives)
    out[8] = P.lin_invA;
    out[9] = P.lin_norange ? P.lin_offA : P.lin_offA1;
    out[10] = P.lin_thrA;
    out[11] = P.lin_nB;
    out[12] = P.lin_mA;
    out[13] = P.lin_cB;
    out[14] = P.lin_norange;
    out[15] = P.lin_log;
    out[16] = P.lin_invB2;
    out[17] = P.lin_thrB;
    out[18] = P.lin_mS;
    return PC_OK;
}

// Host-only view of the constants the FP32 kernel of the same count receives.
extern "C" pc_status pc_fp32_floors(const pc_bins *b, const double cell[3], const double lo[3],
                                    const double hi[3], const double L[3], int periodic,
                                    double rmin, double out[32]) {
    if (!b || !cell || !lo || !hi || !out || (periodic && !L))
        return fail(PC_EINVAL, "pc_fp32_floors: bad arguments");
    Geom g;
    memset(&g, 0, sizeof(g));
    g.periodic = periodic ? 1 : 0;
    for (int a = 0; a < 3; ++a) {
        if (!(cell[a] > 0.0) || !std::isfinite(cell[a]) || !std::isfinite(lo[a]) ||
            !std::isfinite(hi[a]) || hi[a] < lo[a])
            return fail(PC_EINVAL, "pc_fp32_floors: bad cell sides or bounds");
        if (periodic && (!(L[a] > 0.0) || !std::isfinite(L[a])))
            return fail(PC_EINVAL, "pc_fp32_floors: periodic box needs L > 0");
        g.c[a] = cell[a];
        g.c32[a] = (float)cell[a];
        g.ng[a] = 1;
        g.lo[a] = lo[a];
        g.L[a] = periodic ? L[a] : 0.0;
        g.hL[a] = 0.5 * g.L[a];
    }
    Plan P;
    pc_status s = make_plan(b, g, lo, hi, rmin, false, P, false);
    if (s != PC_OK) return s;
    PairParams p;
    memset(static_cast<void *>(&p), 0, sizeof(p));
    p.mode = P.mode;
    p.los = P.los;
    p.n_a = P.na;
    p.n_b = P.nb;
    set_fp32_params(g, lo, hi, P, P.fp32_ok ? PC_PREC_F32_RESCUE : PC_PREC_F64, p);
    const double v[32] = {(double)p.path, (double)p.fix, p.f_inv, p.f_invB, p.f_cfs.x, (double)p.f_ts2, p.f_cfp,
                          (double)p.f_tp2, p.f_lim, p.f_limB, p.f_mA, p.f_mB, p.f_sf2, p.f_sA, p.f_sC, p.f_se2,
                          p.f_close, p.f_tiny.x, p.far, p.f_gm, p.r2prune, p.q2prune, p.zprune, p.lin_invA,
                          p.lin_offA, p.lin_thrA, p.lin_mS, p.lin_nB, p.lin_mA, p.lin_cB, p.lin_invB2, p.lin_thrB};
    for (int k = 0; k < 32; ++k) out[k] = v[k];
    return PC_OK;
}

// Host-only copy of the lookup tables a count's FP32 path would stage (the
// same plan as pc_fp32_bands).
extern "C" pc_status pc_fp32_tables(const pc_bins *b, const double cell[3], const double lo[3],
                                    const double hi[3], const double L[3], int periodic,
                                    double rmin, float *lut, int max_entries, int *n_entries,
                                    double desc[7]) {
    if (!b || !cell || !lo || !hi || !n_entries || !desc || (periodic && !L) ||
        max_entries < 0 || (max_entries > 0 && !lut))
        return fail(PC_EINVAL, "pc_fp32_tables: bad arguments");
    Geom g;
    memset(&g, 0, sizeof(g));
    g.periodic = periodic ? 1 : 0;
    for (int a = 0; a < 3; ++a) {
        if (!(cell[a] > 0.0) || !std::isfinite(cell[a]) || !std::isfinite(lo[a]) ||
            !std::isfinite(hi[a]) || hi[a] < lo[a])
            return fail(PC_EINVAL, "pc_fp32_tables: bad cell sides or bounds");
        if (periodic && (!(L[a] > 0.0) || !std::isfinite(L[a])))
            return fail(PC_EINVAL, "pc_fp32_tables: periodic box needs L > 0");
        g.c[a] = cell[a];
        g.c32[a] = (float)cell[a];
        g.ng[a] = 1;
        g.lo[a] = lo[a];
        g.L[a] = periodic ? L[a] : 0.0;
        g.hL[a] = 0.5 * g.L[a];
    }
    Plan P;
    pc_status s = make_plan(b, g, lo, hi, rmin, false, P, false);
    if (s != PC_OK) return s;
    *n_entries = (int)P.lut.size();
    desc[0] = P.la.off;
    desc[1] = P.la.T;
    desc[2] = P.la.inv_w;
    desc[3] = P.lb.off;
    desc[4] = P.lb.T;
    desc[5] = P.lb.inv_w;
    desc[6] = P.mu_W;
    if ((int)P.lut.size() > max_entries)
        return fail(PC_EOVERFLOW, "pc_fp32_tables: max_entries too small");
    for (size_t k = 0; k < P.lut.size(); ++k) {
        lut[2 * k] = P.lut[k].x;
        lut[2 * k + 1] = P.lut[k].y;
    }
    return PC_OK;
}

// Cost model of Appendix B.1 (cost = a N_pair + b N_node), specialised to the
// GPU kernel: candidate pairs are charged per thread lane (a block occupies
// NT * 2 lanes however many points its cell holds), and every (block,
// stencil row) visit costs a fixed amount of segment building.
extern "C" double pc_suggest_cell_size(long long n, double volume, double r_max, int mode) {
    (void)mode;
    if (!(r_max > 0.0)) return 1.0;
    if (n <= 1 || !(volume > 0.0)) return r_max;
    const double rho = (double)n / volume;
    const double bi = 2.0 * NT;
    const double a = 1.0, brow = 350.0;   // relative costs (lane-pair, block-row)
    double best = r_max, best_cost = INFINITY;
    for (int k = 2; k <= 64; ++k) {
        double c = r_max * 4.0 / k;   // c from 2 R down to R / 16
        double nc = rho * c * c * c;
        if (nc < 4.0 && k > 2) continue;
        double cells = volume / (c * c * c);
        double blocks_per_cell = std::max(1.0, ceil(nc / bi));
        // stencil cells (half shell) by direct count
        double kk = ceil(r_max / c) + 1;
        double ncand_cells = 0, nrows = 0;
        for (int dz = -(int)kk; dz <= (int)kk; ++dz)
            for (int dy = -(int)kk; dy <= (int)kk; ++dy) {
                double my = std::max(std::abs(dy) - 1, 0) * c, mz = std::max(std::abs(dz) - 1, 0) * c;
                double m2 = my * my + mz * mz;
                if (m2 >= r_max * r_max) continue;
                int rx = 0;
                while (true) {
                    double mx = rx * c;
                    if (mx * mx + m2 < r_max * r_max) ++rx; else break;
                }
                ncand_cells += 2 * rx + 1;
                nrows += 1;
            }
        ncand_cells *= 0.5;
        nrows *= 0.5;
        double lanes = cells * blocks_per_cell * bi;
        double cost = a * lanes * ncand_cells * nc + brow * cells * blocks_per_cell * nrows;
        if (cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

extern "C" const char *pc_strerror(pc_status s) {
    switch (s) {
        case PC_OK: return "success";
        case PC_EINVAL: return "invalid argument";
        case PC_ENOMEM: return "out of memory";
        case PC_ECUDA: return "CUDA error";
        case PC_EOVERFLOW: return "size overflow";
        case PC_ETIMEOUT: return "device wait timed out";
        case PC_EUNSUPPORTED: return "unsupported request";
    }
    return "unknown status";
}

extern "C" const char *pc_last_error(void) { return g_last_error.c_str(); }

extern "C" long long pc_launch_count(void) { return launch_count(); }

extern "C" long long pc_alloc_count(void) { return alloc_count(); }

extern "C" const char *pc_version(void) { return "paircount-gb300 0.1 (sm_103a)"; }

// ---------------------------------------------------------------------------
// Auto counts without device allocation.
//
// For callers that must not allocate device memory at count time: code whose
// device memory is owned by another allocator (a framework's caching
// allocator that holds the whole device), loops that must never hit the
// implicit device synchronisation a cudaMalloc/cudaFree can trigger, and
// processes running at their memory limit.  Every temporary of the count
// lives in one file-scope device array of fixed size instead.
// ---------------------------------------------------------------------------
namespace pc {

// Limits of the fixed scratch array (the call rejects anything larger).
constexpr int NA_MAX_BINS = 16384;        // histogram bins
constexpr int NA_MAX_EDGES = 16385;       // edges per axis
constexpr int NA_MAX_CELLS = 1 << 18;     // cells of the grid
constexpr int NA_MAX_BLOCKS = 1 << 19;    // i-blocks
constexpr int NA_MAX_ROWS = 8192;         // stencil rows
constexpr int NA_MAX_LUT = 2 * (MAX_LUT + 2);

struct NaLayout {
    size_t hist, whist, counters, scalars, tasks, stencil, lut, ea, eb, cnt, off, tot, blocks, total;
};

constexpr size_t na_align(size_t x) { return (x + 255) / 256 * 256; }

constexpr NaLayout na_layout() {
    NaLayout L{};
    size_t o = 0;
    L.hist = o;     o = na_align(o + sizeof(unsigned long long) * NA_MAX_BINS);
    L.whist = o;    o = na_align(o + sizeof(double) * NA_MAX_BINS);
    L.counters = o; o = na_align(o + sizeof(unsigned long long) * 4);
    L.scalars = o;  o = na_align(o + sizeof(int) * 4);
    L.tasks = o;    o = na_align(o + sizeof(TaskDev));
    L.stencil = o;  o = na_align(o + sizeof(int4) * NA_MAX_ROWS);
    L.lut = o;      o = na_align(o + sizeof(float2) * NA_MAX_LUT);
    L.ea = o;       o = na_align(o + sizeof(double) * NA_MAX_EDGES);
    L.eb = o;       o = na_align(o + sizeof(double) * NA_MAX_EDGES);
    L.cnt = o;      o = na_align(o + sizeof(int) * (NA_MAX_CELLS + 1));
    L.off = o;      o = na_align(o + sizeof(int) * (NA_MAX_CELLS + 1));
    L.tot = o;      o = na_align(o + sizeof(int) * (NA_MAX_CELLS / 4096 + 2));
    L.blocks = o;   o = na_align(o + sizeof(Block) * NA_MAX_BLOCKS);
    L.total = o;
    return L;
}

constexpr NaLayout NA = na_layout();

// The scratch array (10.8 MiB).  Every GPU that loads the library holds
// it until the process exits.
static __device__ __align__(256) unsigned char g_count_scratch[NA.total];

// Device address of the scratch array on device `dev`, looked up once per
// device with that device current (the host-side symbol is only a stand-in
// and must never be handed to a kernel).
static unsigned char *scratch_on(int dev) {
    static std::map<int, unsigned char *> addr;
    auto it = addr.find(dev);
    if (it != addr.end()) return it->second;
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_count_scratch);
    if (e != cudaSuccess) {
        cuda_fail(e, "cudaGetSymbolAddress(scratch)");
        return nullptr;
    }
    addr[dev] = (unsigned char *)p;
    return (unsigned char *)p;
}

}  // namespace pc

extern "C" pc_status pc_count_auto_noalloc(const pc_grid *g, const pc_bins *b, const pc_opts *opt,
                                           void *stream, long long *counts, double *wcounts) {
    std::lock_guard<std::mutex> lk(api_mutex());
    if (!g) return fail(PC_EINVAL, "pc_count_auto_noalloc: grid is NULL");
    if (!counts && !wcounts) return fail(PC_EINVAL, "pc_count_auto_noalloc: no output buffer");
    if (wcounts && !g->weighted) return fail(PC_EINVAL, "pc_count_auto_noalloc: grid has no weights");
    int cur = -1;
    PC_CUDA(cudaGetDevice(&cur));
    if (cur != g->device)
        return fail(PC_EINVAL, "pc_count_auto_noalloc: the grid's device must be current");
    cudaStream_t st = (cudaStream_t)stream;
    pc_opts o;
    memset(&o, 0, sizeof(o));
    o.priv = -1;
    if (opt) o = *opt;

    if (o.shard_count > 1 && (o.shard_index < 0 || o.shard_index >= o.shard_count))
        return fail(PC_EINVAL, "opts: shard_index must lie in [0, shard_count)");
    Plan P;
    pc_status s = make_plan(b, g->g, g->pts_lo, g->pts_hi, grid_rmin(g), true, P);
    if (s != PC_OK) return s;
    int prec = o.prec;
    if (prec == PC_PREC_F32_RESCUE && !P.fp32_ok) prec = PC_PREC_F64;
    int ipt = (o.ipt == 4) ? 4 : 2;
    if (prec == PC_PREC_F64) ipt = 1;
    const int bi = NT * ipt;
    const long long nblk = (long long)g->ncell + g->n / bi + 16;
    if (P.nbins > NA_MAX_BINS || P.na + 1 > NA_MAX_EDGES || P.nb + 1 > NA_MAX_EDGES)
        return fail(PC_EOVERFLOW, "pc_count_auto_noalloc: more than 16384 bins");
    if (g->ncell > NA_MAX_CELLS)
        return fail(PC_EOVERFLOW, "pc_count_auto_noalloc: grid has more than 262144 cells");
    if (nblk > NA_MAX_BLOCKS)
        return fail(PC_EOVERFLOW, "pc_count_auto_noalloc: more than 524288 point blocks");
    if ((int)P.stencil.size() > NA_MAX_ROWS)
        return fail(PC_EOVERFLOW, "pc_count_auto_noalloc: stencil has more than 8192 rows");
    if ((int)P.lut.size() > NA_MAX_LUT)
        return fail(PC_EOVERFLOW, "pc_count_auto_noalloc: lookup tables too large");

    unsigned char *base = scratch_on(cur);
    if (!base) return PC_ECUDA;
    unsigned long long *hist = (unsigned long long *)(base + NA.hist);
    double *whist = (double *)(base + NA.whist);
    unsigned long long *ctr = (unsigned long long *)(base + NA.counters);
    int *sc = (int *)(base + NA.scalars);
    TaskDev *tasks = (TaskDev *)(base + NA.tasks);

    // everything that must start at zero is cleared on every call
    const size_t hist_n = (size_t)P.nbins;
    PC_CUDA(cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * hist_n, st));
    if (wcounts) PC_CUDA(cudaMemsetAsync(whist, 0, sizeof(double) * hist_n, st));
    PC_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned long long) * 4, st));
    PC_CUDA(cudaMemsetAsync(sc, 0, sizeof(int) * 4, st));
    TaskDev t = task_of(g, g, 0, 1);
    PC_CUDA(cudaMemcpyAsync(tasks, &t, sizeof(TaskDev), cudaMemcpyHostToDevice, st));
    if (!P.stencil.empty())
        PC_CUDA(cudaMemcpyAsync(base + NA.stencil, P.stencil.data(), sizeof(int4) * P.stencil.size(),
                                cudaMemcpyHostToDevice, st));
    if (!P.lut.empty())
        PC_CUDA(cudaMemcpyAsync(base + NA.lut, P.lut.data(), sizeof(float2) * P.lut.size(),
                                cudaMemcpyHostToDevice, st));
    PC_CUDA(cudaMemcpyAsync(base + NA.ea, P.Ea.data(), sizeof(double) * (P.na + 1),
                            cudaMemcpyHostToDevice, st));
    PC_CUDA(cudaMemcpyAsync(base + NA.eb, P.Eb.data(), sizeof(double) * (P.nb + 1),
                            cudaMemcpyHostToDevice, st));
    PC_CUDA(make_blocks_into(tasks, 1, g->ncell, bi, o.shard_count > 1 ? o.shard_index : 0,
                             o.shard_count > 1 ? o.shard_count : 1, (Block *)(base + NA.blocks), sc + 1,
                             (int *)(base + NA.cnt), (int *)(base + NA.off),
                             (int *)(base + NA.tot), st));

    PairParams p;
    memset(static_cast<void *>(&p), 0, sizeof(p));
    p.tasks = tasks;
    p.blocks = (const Block *)(base + NA.blocks);
    p.nblocks = sc + 1;
    p.work_counter = sc;
    p.g = g->g;
    p.stencil = (const int4 *)(base + NA.stencil);
    p.nrows = (int)P.stencil.size();
    p.mode = P.mode;
    p.los = P.los;
    p.weighted = wcounts ? 1 : 0;
    p.n_a = P.na;
    p.n_b = P.nb;
    p.nbins = P.nbins;
    p.r2cut = P.r2cut;
    p.lut = (const float2 *)(base + NA.lut);
    p.lut_total = (int)P.lut.size();
    p.la = P.la;
    p.lb = P.lb;
    p.eps_a = P.eps_a;
    p.eps_b = P.eps_b;
    p.mu_A = P.mu_A;
    p.mu_B = P.mu_B;
    p.mu_W = P.mu_W;
    p.Ea = (const double *)(base + NA.ea);
    p.Eb = (const double *)(base + NA.eb);
    p.hist = hist;
    p.whist = wcounts ? whist : nullptr;
    p.qcount = ctr + 2;
    p.qcap = 0;   // near-edge pairs are checked inside the pair kernel
    p.counters = ctr;
    p.shard_count = o.shard_count > 1 ? o.shard_count : 1;
    p.shard_index = o.shard_count > 1 ? o.shard_index : 0;
    set_fp32_params(g->g, g->pts_lo, g->pts_hi, P, prec, p);
    p.nsub = (bi + 63) / 64;
    p.npts_i = g->n / p.shard_count;
    int sms = 0, per_sm = 0;
    size_t smem = 0;
    PC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, cur));
    // binary64 weight sums here (the exact sums of integer products would need an allocation)
    s = fit_params(prec, o.priv, cur, wcounts != nullptr, false, false, p, smem, per_sm);
    if (s != PC_OK) return s;
    if (per_sm <= 0) return fail(PC_ECUDA, "pair kernel cannot be resident");
    if (o.grid_ctas_per_sm > 0) per_sm = std::min(per_sm, o.grid_ctas_per_sm);
    cudaError_t e = (prec == PC_PREC_F64) ? launch_pairs_f64(p, sms * per_sm, smem, st)
                                          : launch_pairs_f32(p, sms * per_sm, smem, st);
    if (e != cudaSuccess) return cuda_fail(e, "pair kernel launch");
    if (counts) {
        cudaMemcpyKind k = is_device_ptr(counts) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
        PC_CUDA(cudaMemcpyAsync(counts, hist, sizeof(long long) * hist_n, k, st));
    }
    if (wcounts) {
        cudaMemcpyKind k = is_device_ptr(wcounts) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
        PC_CUDA(cudaMemcpyAsync(wcounts, whist, sizeof(double) * hist_n, k, st));
    }
    PC_CUDA(cudaStreamSynchronize(st));
    return PC_OK;
}
