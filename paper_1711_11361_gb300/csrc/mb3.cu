// Three-dimensional moving-boundary cut-cell sweep (Sec. II.C.4, eqs.
// Klein2DcompleteMovingMethod2a-c) for one convex polyhedral body in
// translation, FP64.  One simulation, its own stream; per sweep a fixed
// sequence of kernels over the body's region R (the cells meeting the
// body's bounding box at the sweep's two poses, widened by two cells) and
// over all cells and faces:
//   k3_cells  volume fractions at poses A, M, B and the touch flags (R)
//   k3_faces  apertures at M of the x-, y- and z-faces, time-averaged
//             apertures of the sweep's faces (R)
//   k3_wall   flux-GCL provisional states, shielded distance, wall normal,
//             wall state and flux of the band cells (R)
//   k3_row, k3_march  MUSCL-Hancock states, HLLC + stabilised fluxes and the
//             conservative update alpha_B Q' of every cell: the cells away
//             from R beside the geometry, the others after k3_wall
//   k3_events covering / uncovering, gathered per cell in cell order (R)
//   k3_bad / k3_mix  the positivity safeguard (one block merges in shared memory)
//   k3_final  Q = content / alpha_B in R, solid cells NaN, error checks
//             (elsewhere the content is the state)
// Geometry: the volume of a box inside the body by the divergence theorem
// over the faces of box ∩ body, each face the plane's polygon clipped by all
// other half-spaces in its own plane; apertures by clipping the face
// rectangle.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "mb3.h"
#include "mb3_near.h"
#include "mb_fp64.cuh"

namespace mb3 {

using namespace mbfp;

constexpr int NC = 5;
constexpr int MAXP = MB3_MAX_PLANES;
static_assert(MAXP <= 32, "one plane per lane and per mask bit");
constexpr int MAXH = 6 + MAXP;          // half-spaces of a box inside the body
constexpr int MAXPV = MAXH + 4;         // polygon vertices
constexpr double ALPHA_MIN = 1e-10;
constexpr double COLLAPSE = 0.01;
constexpr int MIX_LAYERS = 8;
constexpr int SEEDCAP = 4096;           // safeguard seeds per sweep
constexpr int NODECAP = 1 << 16;        // safeguard nodes per merge

constexpr int E_UNSTABLE = 1, E_NONBR = 2, E_SEEDCAP = 4, E_NODECAP = 8;

struct Body3 {
    int np;
    double n[3 * MAXP];
    double c[MAXP];     // offsets of the posed planes
    float nf[3 * MAXP], cf[MAXP];   // the same in FP32 (side_of only)
};

// The box [lo, lo + h] (FP32, h >= 0, |lo| + h formed from terms of magnitude
// up to big) against plane f: 1 it lies outside, -1 it lies inside, 0 not
// decided.  Every FP64 corner's distance differs from its FP32 value by less
// than the margin (the rounding of the inputs and of the sums is below 12 x
// 2^-24 of the terms' magnitudes, the margin 4e-6 of them), so a decision is
// the FP64 tests' too.  Most of R is decided so, off the FP64 pipe (44 x 44 x
// 24 cells, two poses: 672 us per launch with FP64 tests, 407 to 468 so; 9.9 M
// FP64 warp instructions against 4.7 M).
__device__ __forceinline__ int side_of(const Body3 &B, int f, const float *lo, const float *h, const float *big) {
    float c = B.cf[f], least = 0.0f, most = 0.0f, mag = fabsf(c);
    for (int a = 0; a < 3; ++a) {
        const float n = B.nf[3 * f + a], e = n * h[a];
        c -= n * lo[a];
        least += fminf(e, 0.0f);
        most += fmaxf(e, 0.0f);
        mag += fabsf(n) * big[a];
    }
    const float m = 4e-6f * mag;
    return least - c > m ? 1 : most - c < -m ? -1 : 0;
}

__host__ __device__ inline double dot3(const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

// area of {p : p = o + s e1 + t e2} clipped by the half-spaces a_m s + b_m t
// <= r_m, starting from the square [-L, L]^2 (a 2-D Sutherland-Hodgman)
// (each vertex's signed distance is evaluated once per half-plane, and a
// half-plane holding every vertex leaves the polygon as it is)
__device__ double clipped_area(const double *a, const double *b, const double *r, int nh, double L) {
    double px[MAXPV], py[MAXPV], qx[MAXPV], qy[MAXPV], s[MAXPV];
    int n = 4;
    px[0] = -L; py[0] = -L; px[1] = L; py[1] = -L; px[2] = L; py[2] = L; px[3] = -L; py[3] = L;
    for (int m = 0; m < nh && n > 0; ++m) {
        bool out = false;
        for (int k = 0; k < n; ++k) {
            s[k] = a[m] * px[k] + b[m] * py[k] - r[m];
            if (!(s[k] <= 0.0)) out = true;
        }
        if (!out) continue;
        int k2 = 0;
        for (int k = 0; k < n; ++k) {
            const int k1 = k + 1 < n ? k + 1 : 0;
            const double sa = s[k], sb = s[k1];
            const bool ina = sa <= 0.0, inb = sb <= 0.0;
            if (ina && k2 < MAXPV) { qx[k2] = px[k]; qy[k2] = py[k]; ++k2; }
            if (ina != inb && k2 < MAXPV) {
                const double t = sa / (sa - sb);
                qx[k2] = px[k] + t * (px[k1] - px[k]);
                qy[k2] = py[k] + t * (py[k1] - py[k]);
                ++k2;
            }
        }
        n = k2;
        for (int k = 0; k < n; ++k) { px[k] = qx[k]; py[k] = qy[k]; }
    }
    if (n < 3) return 0.0;
    double A = 0.0;
    for (int k = 0; k < n; ++k) {
        const int k1 = k + 1 < n ? k + 1 : 0;
        A += px[k] * py[k1] - px[k1] * py[k];
    }
    return 0.5 * A;
}

// volume of the box [lo, lo + h] inside the body; *touch: the body
// boundary cuts the box.  Coordinates relative to lo.  V = (1/3) sum over
// the faces of box ∩ body of offset x area (divergence theorem).  Called by
// all 32 lanes of a warp for the same box: lane l takes faces l, l + 32;
// the sums are reduced over the warp (every exit depends on the box only).
__device__ double box_solid_volume(const Body3 &B, const double *lo, const double *h, bool *touch) {
    const int lane = threadIdx.x & 31;
    double hn[MAXH][3], hc[MAXH];
    int nh = 0;
    for (int a = 0; a < 3; ++a) {   // the box: -x_a <= 0, x_a <= h_a
        for (int s = 0; s < 2; ++s) {
            hn[nh][0] = hn[nh][1] = hn[nh][2] = 0.0;
            hn[nh][a] = s ? 1.0 : -1.0;
            hc[nh] = s ? h[a] : 0.0;
            ++nh;
        }
    }
    const int nbox = nh;
    // the body's planes against the box, lane f taking plane f: over the
    // box's vertices v, n . v is least at v_a = h_a where n_a < 0 (else 0)
    // and greatest at v_a = h_a where n_a > 0, and the rounded sums keep
    // that order; the box lies outside plane f when its lowest vertex does,
    // and plane f cuts it when its highest vertex lies outside
    bool outside = false, cuts = false;
    if (lane < B.np) {
        const double *n = &B.n[3 * lane];
        const double c = B.c[lane] - dot3(n, lo);
        const double vl[3] = {n[0] < 0.0 ? h[0] : 0.0, n[1] < 0.0 ? h[1] : 0.0, n[2] < 0.0 ? h[2] : 0.0};
        const double vh[3] = {n[0] > 0.0 ? h[0] : 0.0, n[1] > 0.0 ? h[1] : 0.0, n[2] > 0.0 ? h[2] : 0.0};
        outside = !(dot3(n, vl) <= c);
        cuts = !outside && !(dot3(n, vh) <= c);
    }
    if (__ballot_sync(0xffffffffu, outside)) { *touch = false; return 0.0; }
    for (unsigned m = __ballot_sync(0xffffffffu, cuts); m; m &= m - 1) {   // the cutting planes in order
        const int f = __ffs(m) - 1;
        const double *n = &B.n[3 * f];
        hn[nh][0] = n[0]; hn[nh][1] = n[1]; hn[nh][2] = n[2];
        hc[nh] = B.c[f] - dot3(n, lo);
        ++nh;
    }
    const double vol = h[0] * h[1] * h[2];
    if (nh == nbox) { *touch = false; return vol; }
    // half-width of the starting square: the polygon of box ∩ plane lies
    // within |h| + |c| of the plane's origin c n
    const double L = 2.0 * sqrt(h[0] * h[0] + h[1] * h[1] + h[2] * h[2]);
    double V = 0.0, body_area = 0.0;
    for (int f = lane; f < nh; f += 32) {
        // in-plane basis e1, e2 (e1 x e2 = n), origin o = c n
        const double *n = hn[f];
        double t[3] = {1.0, 0.0, 0.0};
        if (fabs(n[0]) > 0.9) { t[0] = 0.0; t[1] = 1.0; }
        double e1[3] = {n[1] * t[2] - n[2] * t[1], n[2] * t[0] - n[0] * t[2], n[0] * t[1] - n[1] * t[0]};
        const double l1 = sqrt(dot3(e1, e1));
        for (int q = 0; q < 3; ++q) e1[q] /= l1;
        const double e2[3] = {n[1] * e1[2] - n[2] * e1[1], n[2] * e1[0] - n[0] * e1[2], n[0] * e1[1] - n[1] * e1[0]};
        const double o[3] = {hc[f] * n[0], hc[f] * n[1], hc[f] * n[2]};
        double a[MAXH], b[MAXH], r[MAXH];
        int m2 = 0;
        for (int m = 0; m < nh; ++m) {
            if (m == f) continue;
            a[m2] = dot3(hn[m], e1);
            b[m2] = dot3(hn[m], e2);
            r[m2] = hc[m] - dot3(hn[m], o);
            ++m2;
        }
        const double A = clipped_area(a, b, r, m2, L + fabs(hc[f]));
        V += hc[f] * A;
        if (f >= nbox) body_area += A;
    }
    for (int o = 16; o > 0; o >>= 1) {
        V += __shfl_xor_sync(0xffffffffu, V, o);
        body_area += __shfl_xor_sync(0xffffffffu, body_area, o);
    }
    *touch = body_area > 0.0;
    return fmin(vol, fmax(0.0, V / 3.0));
}

// all 32 lanes of a warp: 1 the box lies outside the body, -1 inside, 0 not
// decided by FP32
__device__ __forceinline__ int box_side(const Body3 &B, const float *lo, const float *h, const float *big) {
    const int lane = threadIdx.x & 31;
    const int s = lane < B.np ? side_of(B, lane, lo, h, big) : -1;
    if (__any_sync(0xffffffffu, s > 0)) return 1;
    return __all_sync(0xffffffffu, s < 0) ? -1 : 0;
}

// solid area of the rectangle {x_a = v} x [lb, lb + wb] x [lc, lc + wc]
// (b, c the axes after a, cyclically): the rectangle clipped by the body's
// planes, in coordinates relative to (lb, lc)
__device__ double rect_solid_area(const Body3 &B, int a, double v, double lb, double wb, double lc, double wc) {
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    // the planes against the rectangle's corners first: none inside one
    // plane leaves no solid, all inside one leaves that plane out
    // (first in FP32, as side_of, which decides most planes)
    unsigned cut = 0, test = 0;
    const float fv = (float)v, fb = (float)lb, fc = (float)lc, hb = (float)wb, hc = (float)wc;
    const float sv = fabsf(fv), sb = fabsf(fb) + hb, sc = fabsf(fc) + hc;
    for (int f = 0; f < B.np; ++f) {
        const float na = B.nf[3 * f + a], nb = B.nf[3 * f + b], nc = B.nf[3 * f + c];
        const float d = B.cf[f] - na * fv - nb * fb - nc * fc, eb = nb * hb, ec = nc * hc;
        const float m = 4e-6f * (fabsf(B.cf[f]) + fabsf(na) * sv + fabsf(nb) * sb + fabsf(nc) * sc);
        if (fminf(eb, 0.0f) + fminf(ec, 0.0f) - d > m) return 0.0;
        if (!(fmaxf(eb, 0.0f) + fmaxf(ec, 0.0f) - d < -m)) test |= 1u << f;
    }
    for (; test; test &= test - 1) {
        const int f = __ffs(test) - 1;
        const double *nn = &B.n[3 * f];
        const double cc = B.c[f] - nn[a] * v - nn[b] * lb - nn[c] * lc;
        const double lo_ = (nn[b] < 0.0 ? nn[b] * wb : 0.0) + (nn[c] < 0.0 ? nn[c] * wc : 0.0) - cc;
        const double hi_ = (nn[b] > 0.0 ? nn[b] * wb : 0.0) + (nn[c] > 0.0 ? nn[c] * wc : 0.0) - cc;
        if (lo_ > 0.0) return 0.0;
        if (hi_ > 0.0) cut |= 1u << f;
    }
    double px[MAXPV], py[MAXPV], qx[MAXPV], qy[MAXPV], s[MAXPV];
    int n = 4;
    px[0] = 0.0; py[0] = 0.0; px[1] = wb; py[1] = 0.0; px[2] = wb; py[2] = wc; px[3] = 0.0; py[3] = wc;
    for (; cut && n > 0; cut &= cut - 1) {
        const int f = __ffs(cut) - 1;
        const double *nn = &B.n[3 * f];
        const double cc = B.c[f] - nn[a] * v - nn[b] * lb - nn[c] * lc;
        bool out = false;   // (as in clipped_area)
        for (int k = 0; k < n; ++k) {
            s[k] = nn[b] * px[k] + nn[c] * py[k] - cc;
            if (!(s[k] <= 0.0)) out = true;
        }
        if (!out) continue;
        int k2 = 0;
        for (int k = 0; k < n; ++k) {
            const int k1 = k + 1 < n ? k + 1 : 0;
            const double sa = s[k], sb = s[k1];
            const bool ina = sa <= 0.0, inb = sb <= 0.0;
            if (ina && k2 < MAXPV) { qx[k2] = px[k]; qy[k2] = py[k]; ++k2; }
            if (ina != inb && k2 < MAXPV) {
                const double t = sa / (sa - sb);
                qx[k2] = px[k] + t * (px[k1] - px[k]);
                qy[k2] = py[k] + t * (py[k1] - py[k]);
                ++k2;
            }
        }
        n = k2;
        for (int k = 0; k < n; ++k) { px[k] = qx[k]; py[k] = qy[k]; }
    }
    if (n < 3) return 0.0;
    double A = 0.0;
    for (int k = 0; k < n; ++k) {
        const int k1 = k + 1 < n ? k + 1 : 0;
        A += px[k] * py[k1] - px[k1] * py[k];
    }
    return fmin(wb * wc, fmax(0.0, 0.5 * A));
}

// ---------------------------------------------------------------------------
// device descriptor: the grid, the region R and the buffers
// ---------------------------------------------------------------------------
struct Desc {
    int nx, ny, nz, n;
    double lo[3], h[3];
    float lof[3], hf[3];    // the same in FP32 (side_of only)
    float bigf[3];          // |lo| + the extent + a cell: bounds every coordinate formed
    int bc[6];
    double gamma, g1h, U[3];   // g1h: (gamma - 1) / 2
    int gcl;
    int d;                  // the sweep's direction
    double lam, hlam;       // dt / h_d and its half
    int r0[3], rn[3];       // region R: first cell and extent per axis
    double *Q, *Qn;         // the state at the sweep's and at the step's start
    double *C;              // contents before the events (R; alpha on its way out of mb3_read_state)
    double *Cn;             // new contents, then the new state
    int f32;                // FP32 flux option
    float *Qf, *Qfn;        // Q and the new state in FP32 (FP32 flux option)
    float gammaf, hlamf;    // gamma and lam / 2 in FP32 (no conversion per thread)
    double *aA, *aM, *aB;   // over R
    unsigned char *tA, *tB; // over R
    double *aP;             // alpha at the sweep's pose A over the region P
    unsigned char *tP;      // (the previous sweep's R), with its touch flags
    int p0[3], pn[3];
    double *bM[3];          // mid-pose apertures of R's faces, per axis
    double *bt;             // time-averaged apertures of R's d-faces
    unsigned char *whas;    // wall data over R
    double *wdist, *wFB, *wQB;
    unsigned char *evt;     // event type over R: 0 none, 1 covered, 2 uncovered donor, 3 covered, leaves
    unsigned *emask;        // recipients / donors (bit (dk+1)*9 + (dj+1)*3 + (di+1))
    double *easum;
    unsigned char *upd;     // over R: the cell has a new content (elsewhere every cell has)
    int *err;
    double *wall;           // 5 summed wall terms
    int *seeds, *nseed;
    int *lab, *par_;        // full grid, -1 where no node (safeguard)
    int *nodes;
    double *ntot;           // (NC + 1) per node
    int *mixed;
    double *smax;           // 3 wave speed maxima (CFL)
};

__device__ __forceinline__ int cidx(const Desc &D, int i, int j, int k) { return (k * D.ny + j) * D.nx + i; }
__device__ __forceinline__ bool in_r(const Desc &D, int i, int j, int k) {
    return i >= D.r0[0] && i < D.r0[0] + D.rn[0] && j >= D.r0[1] && j < D.r0[1] + D.rn[1] && k >= D.r0[2] &&
           k < D.r0[2] + D.rn[2];
}
__device__ __forceinline__ int ridx(const Desc &D, int i, int j, int k) {
    return ((k - D.r0[2]) * D.rn[1] + (j - D.r0[1])) * D.rn[0] + (i - D.r0[0]);
}
// the low a-face of cell (i, j, k) in R's face array of axis a (the cell's
// index along a may be r0 + rn: the high face of R's last cell)
__device__ __forceinline__ bool in_rf(const Desc &D, int a, int i, int j, int k) {
    const int ijk[3] = {i, j, k};
    for (int q = 0; q < 3; ++q) {
        const int hi = D.r0[q] + D.rn[q] + (q == a ? 1 : 0);
        if (ijk[q] < D.r0[q] || ijk[q] >= hi) return false;
    }
    return true;
}
__device__ __forceinline__ int rfidx(const Desc &D, int a, int i, int j, int k) {
    const int m0 = D.rn[0] + (a == 0), m1 = D.rn[1] + (a == 1);
    return ((k - D.r0[2]) * m1 + (j - D.r0[1])) * m0 + (i - D.r0[0]);
}
__device__ __forceinline__ double alphaA(const Desc &D, int i, int j, int k) {
    return in_r(D, i, j, k) ? D.aA[ridx(D, i, j, k)] : 1.0;
}
__device__ __forceinline__ double alphaB(const Desc &D, int i, int j, int k) {
    return in_r(D, i, j, k) ? D.aB[ridx(D, i, j, k)] : 1.0;
}
__device__ __forceinline__ bool updated(const Desc &D, int i, int j, int k) {
    return !in_r(D, i, j, k) || D.upd[ridx(D, i, j, k)];
}
__device__ __forceinline__ double swept(const Desc &D, int i, int j, int k) {
    return in_rf(D, D.d, i, j, k) ? D.bt[rfidx(D, D.d, i, j, k)] : 1.0;
}
// (outside R without a floating-point test: alpha_A = 1 there)
__device__ __forceinline__ bool fluid_a(const Desc &D, int i, int j, int k) {
    if (!in_r(D, i, j, k)) return true;
    const int r = ridx(D, i, j, k);
    const double a = D.aA[r];
    return a > 0.0 || (D.gcl && a == 0.0 && D.aB[r] > 0.0);
}
// float to double exactly by moving the bit fields: integer work, off
// GB300's narrow FP64 pipe, which takes conversions too.  Normal numbers
// rebias the exponent (127 -> 1023); a subnormal m 2^-149 is normalised
// at its highest set bit p; infinities and NaN keep an all-ones exponent
// and the shifted payload
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    const unsigned long long s = (unsigned long long)(u >> 31) << 63;
    unsigned long long b;
    if (e == 0u) {
        if (m == 0u) {
            b = s;
        } else {
            const int p = 31 - __clz((int)m);
            b = s | ((unsigned long long)(p + 874) << 52) | (((unsigned long long)m << (52 - p)) & 0xfffffffffffffULL);
        }
    } else if (e == 0xffu) {
        b = s | (0x7ffULL << 52) | ((unsigned long long)m << 29);
    } else {
        b = s | ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)m << 29);
    }
    return __longlong_as_double((long long)b);
}
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double node(const Desc &D, int a, int i) { return D.lo[a] + (double)i * D.h[a]; }
// x is neither infinite nor NaN: its exponent field is not all ones (an
// integer test, off GB300's narrow FP64 pipe)
__device__ __forceinline__ bool isnan64(double x) {
    return ((unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool finite64(double x) {
    return (__double_as_longlong(x) & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
}

// the state content / alpha_B is physical iff the content is (alpha_B > 0):
// rho > 0 and 2 rho E > |m|^2, no division
__device__ __forceinline__ bool content_bad(const double *q) {
    bool bad = false;
    for (int m = 0; m < NC; ++m) if (!finite64(q[m])) bad = true;   // alpha_B >= 1e-10: the quotient is finite with it
    return bad || !(q[0] > 0.0) || !(2.0 * q[0] * q[4] > q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
}
__device__ __forceinline__ void add_seed(const Desc &D, int c) {
    const int s = atomicAdd(D.nseed, 1);
    if (s < SEEDCAP) D.seeds[s] = c;
    else atomicOr(D.err, E_SEEDCAP);
}
// neighbour (i+di, j+dj, k+dk) under the periodic sides, -1 outside
__device__ __forceinline__ int nbr(const Desc &D, int i, int j, int k, int di, int dj, int dk, int *ii, int *jj,
                                   int *kk) {
    int a = i + di, b = j + dj, c = k + dk;
    if (D.bc[0] == MB_BC_PERIODIC) { a %= D.nx; if (a < 0) a += D.nx; }
    if (D.bc[2] == MB_BC_PERIODIC) { b %= D.ny; if (b < 0) b += D.ny; }
    if (D.bc[4] == MB_BC_PERIODIC) { c %= D.nz; if (c < 0) c += D.nz; }
    if (a < 0 || a >= D.nx || b < 0 || b >= D.ny || c < 0 || c >= D.nz) return -1;
    *ii = a; *jj = b; *kk = c;
    return cidx(D, a, b, c);
}

__device__ __forceinline__ void r_cell(const Desc &D, int t, int *i, int *j, int *k) {
    *i = D.r0[0] + t % D.rn[0];
    *j = D.r0[1] + (t / D.rn[0]) % D.rn[1];
    *k = D.r0[2] + t / (D.rn[0] * D.rn[1]);
}

// the item of a warp-per-item kernel: item v * gridDim.x + b for warp v of
// block b, so that neighbouring items (cut cells cluster along the body's
// surface) land on different blocks, and so on different SMs
__device__ __forceinline__ int warp_item() { return (int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x; }

// volume fractions at the three poses and the touch flags of R's cells,
// one warp per cell and pose (pose B first, then M, then A, so that a
// costly cell's poses run side by side).  CELLS_ALL: poses A, M and B;
// CELLS_REUSE_A: pose A is the previous sweep's pose B, whose values P
// holds (a cell outside P lies two cells or more from the body's bounding
// box: alpha 1, no touch, as computing it gives), copied by the pose-B
// warp; CELLS_ONE: pose B only, into all three
enum { CELLS_ALL = 0, CELLS_REUSE_A = 1, CELLS_ONE = 2 };
__device__ __forceinline__ double fraction(double V, double vol) {
    const double a = fmin(1.0, fmax(0.0, 1.0 - V / vol));
    return a < ALPHA_MIN ? 0.0 : a;
}
__global__ void k3_cells(Desc D, Body3 BA, Body3 BM, Body3 BB, int mode) {
    const int rc = D.rn[0] * D.rn[1] * D.rn[2];
    const int w = warp_item();
    const int npose = mode == CELLS_ALL ? 3 : mode == CELLS_REUSE_A ? 2 : 1;
    if (w >= npose * rc) return;
    const int t = w % rc, pose = w / rc;   // 0: B, 1: M, 2: A
    int i, j, k;
    r_cell(D, t, &i, &j, &k);
    const Body3 &B = pose == 0 ? BB : pose == 1 ? BM : BA;
    const float fl[3] = {D.lof[0] + i * D.hf[0], D.lof[1] + j * D.hf[1], D.lof[2] + k * D.hf[2]};
    const int side = box_side(B, fl, D.hf, D.bigf);
    bool touch = false;
    double a = side > 0 ? 1.0 : 0.0;   // no solid, or solid throughout
    if (side == 0) {
        const double lo[3] = {node(D, 0, i), node(D, 1, j), node(D, 2, k)};
        const double hi[3] = {node(D, 0, i + 1), node(D, 1, j + 1), node(D, 2, k + 1)};
        const double h[3] = {hi[0] - lo[0], hi[1] - lo[1], hi[2] - lo[2]};
        a = fraction(box_solid_volume(B, lo, h, &touch), h[0] * h[1] * h[2]);
    }
    if ((threadIdx.x & 31) != 0) return;
    if (pose == 0) {
        D.aB[t] = a;
        D.tB[t] = touch;
        if (mode == CELLS_ONE) {
            D.aM[t] = a;
            D.aA[t] = a;
            D.tA[t] = touch;
        } else if (mode == CELLS_REUSE_A) {
            const bool inP = i >= D.p0[0] && i < D.p0[0] + D.pn[0] && j >= D.p0[1] && j < D.p0[1] + D.pn[1] &&
                             k >= D.p0[2] && k < D.p0[2] + D.pn[2];
            const int q = inP ? ((k - D.p0[2]) * D.pn[1] + (j - D.p0[1])) * D.pn[0] + (i - D.p0[0]) : 0;
            D.aA[t] = inP ? D.aP[q] : 1.0;
            D.tA[t] = inP ? D.tP[q] : 0;
        }
    } else if (pose == 1) {
        D.aM[t] = a;
    } else {
        D.aA[t] = a;
        D.tA[t] = touch;
    }
}

// apertures at M of R's x-, y- and z-faces, then the time-averaged
// apertures of R's d-faces (the fluid fraction of [x_f - delta, x_f] with
// the body at A), one face per thread over the four index ranges
__global__ void k3_faces(Desc D, Body3 BM, Body3 BA, double delta) {
    int t = warp_item() * 32 + (int)(threadIdx.x & 31);   // whole warps spread over blocks
    for (int a = 0; a < 4; ++a) {
        const int ax = a < 3 ? a : D.d;
        const int m0 = D.rn[0] + (ax == 0), m1 = D.rn[1] + (ax == 1), m2 = D.rn[2] + (ax == 2);
        const int cnt = m0 * m1 * m2;
        if (t >= cnt) { t -= cnt; continue; }
        const int ijk[3] = {D.r0[0] + t % m0, D.r0[1] + (t / m0) % m1, D.r0[2] + t / (m0 * m1)};
        const int b = (ax + 1) % 3, c = (ax + 2) % 3;
        if (a < 3) {
            const double lb = node(D, b, ijk[b]), wb = node(D, b, ijk[b] + 1) - lb;
            const double lc = node(D, c, ijk[c]), wc = node(D, c, ijk[c] + 1) - lc;
            const double A = rect_solid_area(BM, ax, node(D, ax, ijk[ax]), lb, wb, lc, wc);
            D.bM[ax][t] = fmin(1.0, fmax(0.0, 1.0 - A / (wb * wc)));
        } else if (delta == 0.0) {
            const double lb = node(D, b, ijk[b]), wb = node(D, b, ijk[b] + 1) - lb;
            const double lc = node(D, c, ijk[c]), wc = node(D, c, ijk[c] + 1) - lc;
            const double A = rect_solid_area(BA, ax, node(D, ax, ijk[ax]), lb, wb, lc, wc);
            D.bt[t] = fmin(1.0, fmax(0.0, 1.0 - A / (wb * wc)));
        }
        return;
    }
}

// time-averaged apertures of R's d-faces for delta != 0: the fluid fraction
// of [x_f - delta, x_f] with the body at A, one warp per face
__global__ void k3_swept(Desc D, Body3 BA, double delta) {
    const int t = warp_item();
    const int ax = D.d;
    const int m0 = D.rn[0] + (ax == 0), m1 = D.rn[1] + (ax == 1), m2 = D.rn[2] + (ax == 2);
    if (t >= m0 * m1 * m2) return;
    const int ijk[3] = {D.r0[0] + t % m0, D.r0[1] + (t / m0) % m1, D.r0[2] + t / (m0 * m1)};
    {
        float fl[3], fh[3], big[3];
        const float dl = (float)delta;
        for (int q = 0; q < 3; ++q) {
            const bool m = q == ax;
            fl[q] = D.lof[q] + ijk[q] * D.hf[q] - (m && dl > 0.0f ? dl : 0.0f);
            fh[q] = m ? fabsf(dl) : D.hf[q];
            big[q] = D.bigf[q] + (m ? fabsf(dl) : 0.0f);
        }
        const int side = box_side(BA, fl, fh, big);
        if (side != 0) {
            if ((threadIdx.x & 31) == 0) D.bt[t] = side > 0 ? 1.0 : 0.0;
            return;
        }
    }
    double lo[3], h[3];
    for (int q = 0; q < 3; ++q) { lo[q] = node(D, q, ijk[q]); h[q] = node(D, q, ijk[q] + 1) - lo[q]; }
    const double xf = node(D, ax, ijk[ax]);
    const double s0 = delta > 0.0 ? xf - delta : xf, s1 = delta > 0.0 ? xf : xf - delta;
    lo[ax] = s0;
    h[ax] = s1 - s0;
    bool tch;
    const double V = box_solid_volume(BA, lo, h, &tch);
    if ((threadIdx.x & 31) == 0) D.bt[t] = fmin(1.0, fmax(0.0, 1.0 - V / (h[0] * h[1] * h[2])));
}

// exact wall Riemann problem (eq. riemann_wallvel), normal n into the body
__device__ void wall_state3(double g, const double *q, const double *n, const double *w, double *rs, double *ps,
                            double *us) {
    const double rho = q[0];
    const double u[3] = {q[1] / rho, q[2] / rho, q[3] / rho};
    const double p = (g - 1.0) * (q[4] - 0.5 * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) / rho);
    const double du = (u[0] * n[0] + u[1] * n[1] + u[2] * n[2]) - (w[0] * n[0] + w[1] * n[1] + w[2] * n[2]);
    const double mu = (g - 1.0) / (g + 1.0);
    double pst, rst;
    if (du > 0.0) {
        const double A = 2.0 / ((g + 1.0) * rho), Bc = mu * p;
        pst = p + du / (2.0 * A) * (du + sqrt(du * du + 4.0 * A * (p + Bc)));
        const double pr = pst / p;
        rst = rho * (pr + mu) / (mu * pr + 1.0);
    } else {
        const double c = sqrt(g * p / rho);
        const double x = 1.0 + 0.5 * (g - 1.0) * du / c;
        if (x > 0.0) {
            pst = p * pow(x, 2.0 * g / (g - 1.0));
            rst = rho * pow(pst / p, 1.0 / g);
        } else {
            pst = 0.0;
            rst = 0.0;
        }
    }
    *ps = pst > 1e-12 * p ? pst : 1e-12 * p;
    *rs = rst > 1e-12 * rho ? rst : 1e-12 * rho;
    for (int m = 0; m < 3; ++m) us[m] = u[m] - du * n[m];
}

// flux-GCL provisional states of uncovered cells (in place in Q), then the
// wall data of R's band cells (Sec. II.B, II.C.3, II.C.4)
__global__ void k3_wall(Desc D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= D.rn[0] * D.rn[1] * D.rn[2]) return;
    int i, j, k;
    r_cell(D, t, &i, &j, &k);
    const int c = cidx(D, i, j, k);
    const double aA = D.aA[t], aB = D.aB[t];
    if (D.gcl && aA == 0.0 && aB > 0.0) {
        double acc[NC] = {0, 0, 0, 0, 0}, wsum = 0.0;
        for (int pass = 0; pass < 3 && wsum == 0.0; ++pass)
            for (int dk = -1; dk <= 1; ++dk)
                for (int dj = -1; dj <= 1; ++dj)
                    for (int di = -1; di <= 1; ++di) {
                        const int nzc = (di != 0) + (dj != 0) + (dk != 0);
                        if (nzc == 0 || nzc > pass + 1) continue;
                        int ii, jj, kk;
                        const int cc = nbr(D, i, j, k, di, dj, dk, &ii, &jj, &kk);
                        if (cc < 0) continue;
                        const double w = alphaA(D, ii, jj, kk);
                        if (!(w > 0.0)) continue;
                        wsum += w;
                        for (int q = 0; q < NC; ++q) acc[q] += w * D.Q[(size_t)q * D.n + cc];
                    }
        if (wsum == 0.0) atomicOr(D.err, E_NONBR);
        else for (int q = 0; q < NC; ++q) {
            D.Q[(size_t)q * D.n + c] = acc[q] / wsum;
            if (D.f32) D.Qf[(size_t)q * D.n + c] = float(acc[q] / wsum);
        }
    }
    const bool fl = aA > 0.0 || (D.gcl && aA == 0.0 && aB > 0.0);
    D.whas[t] = 0;
    if (!fl || !(D.tA[t] || D.tB[t])) return;
    const int d = D.d;
    int hi[3] = {i, j, k};
    hi[d] += 1;
    const double blo = D.bM[d][rfidx(D, d, i, j, k)], bhi = D.bM[d][rfidx(D, d, hi[0], hi[1], hi[2])];
    const double db = fabs(blo - bhi);
    const double ahat = D.aM[t] - fmin(blo, bhi);
    D.wdist[t] = db > 1e-12 ? fmin(1.0, fmax(0.0, ahat / db)) : 1.0;
    double nL[3];
    for (int a = 0; a < 3; ++a) {
        int up[3] = {i, j, k};
        up[a] += 1;
        const double bl = D.bM[a][rfidx(D, a, i, j, k)], bu = D.bM[a][rfidx(D, a, up[0], up[1], up[2])];
        nL[a] = (bl - bu) * D.h[(a + 1) % 3] * D.h[(a + 2) % 3];
    }
    const double L = sqrt(nL[0] * nL[0] + nL[1] * nL[1] + nL[2] * nL[2]);
    double nn[3];
    for (int a = 0; a < 3; ++a) nn[a] = L > 0.0 ? nL[a] / L : 0.0;
    double qc[NC], qn[NC];
    const bool fresh = isnan(D.Qn[c]);
    for (int q = 0; q < NC; ++q) {
        qc[q] = D.Q[(size_t)q * D.n + c];
        qn[q] = fresh ? qc[q] : D.Qn[(size_t)q * D.n + c];
    }
    const double g = D.gamma;
    double rs, ps_step, us[3], rs2, ps_sw, us2[3];
    wall_state3(g, qn, nn, D.U, &rs, &ps_step, us);
    wall_state3(g, qc, nn, D.U, &rs2, &ps_sw, us2);
    const double Eadv = ps_step / (g - 1.0) + 0.5 * rs * (us[0] * us[0] + us[1] * us[1] + us[2] * us[2]);
    const double ud = us[d];
    double *FB = &D.wFB[(size_t)NC * t], *QB = &D.wQB[(size_t)NC * t];
    QB[0] = rs;
    for (int m = 0; m < 3; ++m) QB[1 + m] = rs * us[m];
    QB[4] = Eadv;
    FB[0] = rs * ud;
    for (int m = 0; m < 3; ++m) FB[1 + m] = rs * ud * us[m] + (m == d ? ps_sw : 0.0);
    FB[4] = ud * (Eadv + ps_step);
    D.whas[t] = 1;
}

// ---------------------------------------------------------------------------
// fluxes, update, events, safeguard, new states
// ---------------------------------------------------------------------------
__device__ __forceinline__ double pressure5(double g, const double *q) {
    return (g - 1.0) * (q[4] - 0.5 * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) / q[0]);
}
// The line kernels' flow arithmetic in the type T: double for the FP64 path
// (mb_fp64.cuh), float for the FP32 flux option (below; the file is built
// without contraction, so it fuses where it says so).
__device__ __forceinline__ float fmad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float sq3(const float *m) { return fmad(m[0], m[0], fmad(m[1], m[1], m[2] * m[2])); }
// the physical flux along d of a state with 1/rho given
template <int d>
__device__ __forceinline__ void flux5(float g, const float *q, float ir, float *f) {
    const float rho = q[0], un = q[1 + d] * ir;
    const float p = (g - 1.0f) * fmad(-0.5f * sq3(q + 1), ir, q[4]);
    f[0] = rho * un;
    for (int m = 0; m < 3; ++m) f[1 + m] = m == d ? fmad(q[1 + m], un, p) : q[1 + m] * un;
    f[4] = un * (q[4] + p);
}
// HLLC, Davis wave speeds (Toro, Riemann Solvers ch. 10)
template <int d>
__device__ __forceinline__ void hllc5(float g, const float *qL, const float *qR, float *F) {
    constexpr int in = 1 + d;
    // 1/rho of both states from one reciprocal of their product
    const float rL = qL[0], rR = qR[0], rr2 = 1.0f / (rL * rR), iL = rR * rr2, iR = rL * rr2;
    const float uL = qL[in] * iL, uR = qR[in] * iR;
    const float pL = (g - 1.0f) * fmad(-0.5f * sq3(qL + 1), iL, qL[4]);
    const float pR = (g - 1.0f) * fmad(-0.5f * sq3(qR + 1), iR, qR[4]);
    const float cL = sqrtf(g * pL * iL), cR = sqrtf(g * pR * iR);
    const float SL = fminf(uL - cL, uR - cR), SR = fmaxf(uL + cL, uR + cR);
    if (SL >= 0.0f) { flux5<d>(g, qL, iL, F); return; }
    if (SR <= 0.0f) { flux5<d>(g, qR, iR, F); return; }
    const float num = fmad(-(rR * uR), SR - uR, fmad(rL * uL, SL - uL, pR - pL));
    const float den = fmad(rL, SL - uL, -(rR * (SR - uR)));
    const float Ss = num / den;
    const bool left = Ss >= 0.0f;
    float q[NC];
    for (int k = 0; k < NC; ++k) q[k] = left ? qL[k] : qR[k];
    const float r = q[0], ir = left ? iL : iR, u = left ? uL : uR, p = left ? pL : pR;
    const float S = left ? SL : SR;
    float f[NC], qs[NC];
    f[0] = r * u;
    for (int m = 0; m < 3; ++m) f[1 + m] = m == d ? fmad(q[1 + m], u, p) : q[1 + m] * u;
    f[4] = u * (q[4] + p);
    // fac = a / dS and p / a with a = rho (S - u), dS = S - S*, from one
    // reciprocal of a dS
    const float a = r * (S - u), dS = S - Ss, rr = 1.0f / (a * dS);
    const float fac = a * a * rr;
    qs[0] = fac;
    for (int m = 0; m < 3; ++m) qs[1 + m] = m == d ? fac * Ss : fac * (q[1 + m] * ir);
    qs[4] = fac * fmad(q[4], ir, (Ss - u) * fmad(p * dS, rr, Ss));
    for (int k = 0; k < NC; ++k) F[k] = fmad(S, qs[k] - q[k], f[k]);
}
__device__ __forceinline__ float vanleer(float dm, float dp) {
    const float pr = dm * dp;
    return pr > 0.0f ? 2.0f * pr / (dm + dp) : 0.0f;
}

// MUSCL-Hancock evolved boundary states L, R of a cell from its state and its
// neighbours' along d (conserved variables, van Leer, zero slope next to a
// solid cell (!lim), first order where an evolved state is not physical),
// and the HLLC flux of two of them, widened to FP64
template <typename T, int d> struct Flow;
template <int d> struct Flow<double, d> {
    using S = Side<NC>;
    double g, h1, hl;
    __device__ __forceinline__ explicit Flow(const Desc &D) : g(D.gamma), h1(D.g1h), hl(D.hlam) {}
    __device__ __forceinline__ void states(const double *qm, const double *q0, const double *qp, bool lim, S &L,
                                           S &R) const {
        evolve64<NC, d>(h1, hl, qm, q0, qp, lim, L, R);
    }
    __device__ __forceinline__ void flux(const S &L, const S &R, double *F) const { hllc64<NC, d>(g, L, R, F); }
};
template <int d> struct Flow<float, d> {
    struct S { float q[NC]; };
    float g, hl;
    __device__ __forceinline__ explicit Flow(const Desc &D) : g(D.gammaf), hl(D.hlamf) {}
    __device__ __forceinline__ void states(const float *qm, const float *q0, const float *qp, bool lim, S &L,
                                           S &R) const {
        float qL[NC], qR[NC], fL[NC], fR[NC];
        for (int k = 0; k < NC; ++k) {
            const float sl = lim ? vanleer(q0[k] - qm[k], qp[k] - q0[k]) : 0.0f;
            qL[k] = fmad(-0.5f, sl, q0[k]);
            qR[k] = fmad(0.5f, sl, q0[k]);
        }
        const float rr2 = 1.0f / (qL[0] * qR[0]);   // 1/rho of both extrapolated states
        flux5<d>(g, qL, qR[0] * rr2, fL);
        flux5<d>(g, qR, qL[0] * rr2, fR);
        for (int k = 0; k < NC; ++k) {
            const float df = fL[k] - fR[k];
            L.q[k] = fmad(hl, df, qL[k]);
            R.q[k] = fmad(hl, df, qR[k]);
        }
        // physical: rho > 0 and p > 0, i.e. 2 rho E > |m|^2
        auto ok = [](const float *Q) {
            return Q[0] > 0.0f && 2.0f * Q[0] * Q[4] > Q[1] * Q[1] + Q[2] * Q[2] + Q[3] * Q[3];
        };
        if (!ok(L.q) || !ok(R.q))
            for (int k = 0; k < NC; ++k) { L.q[k] = q0[k]; R.q[k] = q0[k]; }
    }
    __device__ __forceinline__ void flux(const S &L, const S &R, float *F) const { hllc5<d>(g, L.q, R.q, F); }
    __device__ __forceinline__ void flux(const S &L, const S &R, double *F) const {
        float f[NC];
        hllc5<d>(g, L.q, R.q, f);
        for (int k = 0; k < NC; ++k) F[k] = widen(f[k]);
    }
};
// the type of a face's flux: FP64 near the body, where it is stabilised
template <typename T, bool GEN> using FluxT = std::conditional_t<GEN, double, T>;
// F_lo - F_hi in FP64 (so that the update's differences telescope as in the
// FP64 path).  FP32 fluxes: where all five FP32 differences are exact (their
// rounding errors by Knuth's two-sum are zero: neighbouring fluxes mostly lie
// within a factor of two) they are widened, else the fluxes are widened and
// subtracted, the same values either way with five FP64 instructions fewer
__device__ __forceinline__ void flux_diff(const double *lo, const double *hi, double *df) {
    for (int k = 0; k < NC; ++k) df[k] = lo[k] - hi[k];
}
__device__ __forceinline__ void flux_diff(const float *lo, const float *hi, double *df) {
    float s[NC];
    bool exact = true;
    for (int k = 0; k < NC; ++k) {
        s[k] = lo[k] - hi[k];
        const float b = s[k] - lo[k];
        exact = exact && (lo[k] - (s[k] - b)) + (-hi[k] - b) == 0.0f;
    }
    if (exact)
        for (int k = 0; k < NC; ++k) df[k] = widen(s[k]);
    else
        for (int k = 0; k < NC; ++k) df[k] = widen(lo[k]) - widen(hi[k]);
}
// the state array of the type T
template <typename T> __device__ __forceinline__ const T *qsrc(const Desc &D);
template <> __device__ __forceinline__ const double *qsrc<double>(const Desc &D) { return D.Q; }
template <> __device__ __forceinline__ const float *qsrc<float>(const Desc &D) { return D.Qf; }
// position m along a line of nal cells with the boundary conditions' ghosts:
// the cell it is or mirrors, *flip for a reflective mirror
__device__ __forceinline__ int line_pos(const Desc &D, int d, int m, int nal, bool *flip) {
    *flip = false;
    if (m >= 0 && m < nal) return m;
    const int bc = D.bc[m < 0 ? 2 * d : 2 * d + 1];
    if (bc == MB_BC_PERIODIC) { m %= nal; return m < 0 ? m + nal : m; }
    *flip = bc == MB_BC_REFLECTIVE;
    return m < 0 ? -1 - m : 2 * nal - 1 - m;
}

// The face f of a line in R's neighbourhood (f the low d-face of cell ijk[d] =
// f, f = nal the high face of the last cell): its HLLC flux becomes the
// stabilised flux bf F2D (eqs. Klein2DtotalfluxaMethod2,
// Klein2shieldedFluxMethod2, with the two-sided shielded parts); both cells
// are fluid and bf > 0
template <typename T, int d>
__device__ __forceinline__ void stabilise(const Desc &D, const int *ijk, int f, int nal, bool periodic, bool fin,
                                          double bf, double *F) {
    const int mR = f < nal ? f : -1, mL = f >= 1 ? f - 1 : (periodic ? nal - 1 : -1);
    double sR = 0.0, sL = 0.0, dR = 0.0, dL = 0.0;
    const double *FBR = nullptr, *FBL = nullptr;
    bool wall = false;   // a neighbour has wall data (else sR = sL = 0)
    int c3[3] = {ijk[0], ijk[1], ijk[2]};
    if (mR >= 0) {
        c3[d] = mR;
        if (in_r(D, c3[0], c3[1], c3[2])) {
            const int r = ridx(D, c3[0], c3[1], c3[2]);
            if (D.whas[r]) {
                wall = true;
                c3[d] = mR + 1 < nal || !periodic ? mR + 1 : 0;
                sR = fmax(0.0, bf - swept(D, c3[0], c3[1], c3[2]));
                dR = D.wdist[r];
                FBR = &D.wFB[(size_t)NC * r];
            }
        }
    }
    if (mL >= 0) {
        c3[d] = mL;
        if (in_r(D, c3[0], c3[1], c3[2])) {
            const int r = ridx(D, c3[0], c3[1], c3[2]);
            if (D.whas[r]) {
                wall = true;
                sL = fmax(0.0, bf - swept(D, c3[0], c3[1], c3[2]));
                dL = D.wdist[r];
                FBL = &D.wFB[(size_t)NC * r];
            }
        }
    }
    if (wall && sR + sL > bf) {
        const double sc = bf / (sR + sL);
        sR *= sc;
        sL *= sc;
    }
    if (wall && (sR > 0.0 || sL > 0.0)) {
        for (int q = 0; q < NC; ++q) {
            const double Fq = F[q];
            double v = (bf - sL - sR) * Fq;
            if (sR > 0.0) v += sR * (FBR[q] + dR * (Fq - FBR[q]));
            if (sL > 0.0) v += sL * (FBL[q] + dL * (Fq - FBL[q]));
            F[q] = v;
        }
    } else if (fin && bf != 1.0) {
        // (the FP32 option's product in FP32)
        for (int q = 0; q < NC; ++q) F[q] = sizeof(T) == 4 ? widen((float)bf * (float)F[q]) : bf * F[q];
    }
}
// flux of face f of the line through ijk between cells with states L (of the
// low cell) and R; GEN: zero next to a solid cell, stabilised near the body
template <typename T, int d, bool GEN>
__device__ __forceinline__ void line_flux(const Desc &D, const Flow<T, d> &fl, const int *line, int f, int nal,
                                          bool fluids, const typename Flow<T, d>::S &L, const typename Flow<T, d>::S &R,
                                          FluxT<T, GEN> *F) {
    if constexpr (GEN) {
        const bool periodic = D.bc[2 * d] == MB_BC_PERIODIC;
        int ijk[3] = {line[0], line[1], line[2]};
        ijk[d] = periodic && f == nal ? 0 : f;
        const bool fin = in_rf(D, d, ijk[0], ijk[1], ijk[2]);
        const double bf = fin ? D.bt[rfidx(D, d, ijk[0], ijk[1], ijk[2])] : 1.0;
        for (int q = 0; q < NC; ++q) F[q] = 0.0;
        if (!fluids || (fin && !(bf > 0.0))) return;
        fl.flux(L, R, F);
        stabilise<T, d>(D, ijk, ijk[d], nal, periodic, fin, bf, F);
    } else {
        fl.flux(L, R, F);
    }
}

// the content update x = Q + lam (F_lo - F_hi) of a cell away from the body
// (fused for the FP64 path; the FP32 option rounds each operation)
__device__ __forceinline__ double content(double lam, double q, double df, double) { return __fma_rn(lam, df, q); }
__device__ __forceinline__ double content(double lam, double q, double df, float) { return q + lam * df; }
// alpha_B Q' = alpha_A Q + lam (F_lo - F_hi) + lam (beta_hi - beta_lo)(F^B -
// w_d Q^B) (eqs. Klein2DcompleteMovingMethod2a-c) of cell m of the line
// through ijk, index c, into Cn (in R also C and upd; elsewhere the FP32 copy
// and the safeguard's seed test: alpha_A = alpha_B = 1 there and no event
// changes the content).  w: this thread's wall terms.
template <typename T, int d, bool GEN>
__device__ __forceinline__ void line_update(const Desc &D, const int *line, int m, int nal, int c, const double *Q,
                                            const FluxT<T, GEN> *Flo, const FluxT<T, GEN> *Fhi, double *w) {
    double v[NC], df[NC];
    flux_diff(Flo, Fhi, df);
    if (GEN) {
        int ijk[3] = {line[0], line[1], line[2]};
        ijk[d] = m;
        if (in_r(D, ijk[0], ijk[1], ijk[2])) {
            const int r = ridx(D, ijk[0], ijk[1], ijk[2]);
            const bool fl = fluid_a(D, ijk[0], ijk[1], ijk[2]);
            const double aA = D.aA[r];
            const double blo = swept(D, ijk[0], ijk[1], ijk[2]);
            ijk[d] = m + 1 < nal || D.bc[2 * d] != MB_BC_PERIODIC ? m + 1 : 0;
            const double bhi = swept(D, ijk[0], ijk[1], ijk[2]);
            const bool wall = fl && D.whas[r] && blo != bhi;
            for (int q = 0; q < NC; ++q) {
                v[q] = 0.0;
                if (fl) v[q] = aA * Q[q] + D.lam * df[q];
                if (wall) {
                    const double wt = D.lam * (bhi - blo) * (D.wFB[(size_t)NC * r + q] -
                                                             D.U[d] * D.wQB[(size_t)NC * r + q]);
                    v[q] += wt;
                    w[q] += wt;
                }
                D.C[(size_t)q * D.n + c] = v[q];
                D.Cn[(size_t)q * D.n + c] = v[q];
            }
            D.upd[r] = fl;
            return;
        }
    }
    for (int q = 0; q < NC; ++q) {
        v[q] = content(D.lam, Q[q], df[q], T(0));
        D.Cn[(size_t)q * D.n + c] = v[q];
    }
    if (sizeof(T) == 4) {
        float x[NC];
        for (int q = 0; q < NC; ++q) {
            x[q] = narrow32(v[q]);
            D.Qfn[(size_t)q * D.n + c] = x[q];
        }
        // the seed test in FP32 where that decides with a margin of 1e-5
        // (and no product underflows)
        const float t = 2.0f * x[0] * x[4];
        if (!(x[0] > 0.0f && x[4] > 0.0f && t > 1e-30f && t < 1e38f && t - sq3(x + 1) > 1e-5f * t) &&
            content_bad(v))
            add_seed(D, c);
    } else if (!physical64<NC>(v)) {
        if (content_bad(v)) add_seed(D, c);
    }
}
// a warp's wall terms, one atomic per component
__device__ __forceinline__ void add_wall(const Desc &D, const double *w) {
    bool any = false;
    for (int q = 0; q < NC; ++q) any = any || w[q] != 0.0;
    if (!__any_sync(0xffffffffu, any)) return;
    for (int q = 0; q < NC; ++q) {
        double s = w[q];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(&D.wall[q], s);
    }
}

// The near cells of a sweep along d: the lines through R's cross-section, from
// two cells before R to two after its last d-face (over a periodic side too).
// Only their update reads body data: k3_row and k3_march update all other
// cells, beside the geometry, and k3_near_row and k3_near the near ones after
// k3_wall (few, and FP64 chains: as many threads as there are cells).
__host__ __device__ inline Near near_range(const Desc &D, int d, int nal) {
    return near_span(D.r0[d], D.rn[d], nal, D.bc[2 * d] == MB_BC_PERIODIC);
}
__device__ __forceinline__ bool near_line(const Desc &D, int d, const int *ijk) {
    bool in = D.rn[0] > 0;
    for (int q = 0; q < 3; ++q) in = in && (q == d || (ijk[q] >= D.r0[q] && ijk[q] < D.r0[q] + D.rn[q]));
    return in;
}

// x sweep.  The line kernels keep the evolved states and the fluxes in
// registers: per cell they read the state and write the new one (80 bytes; 120
// with the FP32 copy), where a kernel each for the states, the fluxes, the
// update and the new state moved 400.  FP64: bound by the FP64 pipe; 4 M cells
// whose states all vary, per sweep, before -> after: x 2520 -> 1265 us, y 2400
// -> 1368, z 2390 -> 1373, 173 lane operations per cell at 0.85 of the pipe's
// rate (uniform states on both sides of a shock take fewer: 153 to 158, 1161 to
// 1225 us).  FP32 option: 12 to 13 FP64 lane operations per cell (the update)
// and 670 to 790 instructions; 32 M cells per sweep, 3790 -> 857 us (x), 1041,
// 1066.  Rows are laid end to end as slots, position -1 .. nx of every row, and
// a warp takes 32 slots from slot 30 w on: it evolves 32 positions, forms 31
// fluxes and updates 30 cells, whatever the row length.
template <typename T, bool GEN>
__device__ __forceinline__ void row_unit(const Desc &D, bool store, int p, int j, int k) {
    const Flow<T, 0> fl(D);
    const int line[3] = {0, j, k};
    const int row = (k * D.ny + j) * D.nx;
    const T *__restrict__ Q = qsrc<T>(D) + row;
    T q[3][NC];
    bool fu[3];
    for (int s = 0; s < 3; ++s) {
        bool flip;
        const int c = line_pos(D, 0, p - 1 + s, D.nx, &flip);
        for (int m = 0; m < NC; ++m) q[s][m] = Q[(size_t)m * D.n + c];
        if (flip) q[s][1] = -q[s][1];
        fu[s] = !GEN || fluid_a(D, c, j, k);
    }
    double Qd[NC];   // the cell's FP64 state
    for (int m = 0; m < NC; ++m)
        Qd[m] = sizeof(T) == 8 ? (double)q[1][m] : store ? D.Q[(size_t)m * D.n + row + p] : 0.0;
    typename Flow<T, 0>::S L, R;
    fl.states(q[0], q[1], q[2], fu[0] && fu[2], L, R);
    {   // the right state of the slot below
        T *x = reinterpret_cast<T *>(&R);
        for (int m = 0; m < (int)(sizeof(R) / sizeof(T)); ++m) x[m] = __shfl_up_sync(0xffffffffu, x[m], 1);
    }
    FluxT<T, GEN> F[NC], Fhi[NC];
    line_flux<T, 0, GEN>(D, fl, line, max(p, 0), D.nx, fu[0] && fu[1], R, L, F);
    for (int m = 0; m < NC; ++m) Fhi[m] = __shfl_down_sync(0xffffffffu, F[m], 1);
    double w[NC] = {0, 0, 0, 0, 0};
    if (store) line_update<T, 0, GEN>(D, line, p, D.nx, row + p, Qd, F, Fhi, w);
    if (GEN) add_wall(D, w);
}
// slot s of rows of len positions: its row, its position in it
__device__ __forceinline__ unsigned row_slot(unsigned len, unsigned *s) {
    *s = (unsigned)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 30u + (threadIdx.x & 31u);
    const unsigned row = *s / len;
    *s -= row * len;
    return row;
}
__device__ __forceinline__ bool mid_lane() { return (threadIdx.x & 31u) - 1u < 30u; }
template <typename T>
__global__ void __launch_bounds__(128, 4) k3_row(Desc D) {
    const unsigned rows = (unsigned)(D.ny * D.nz);
    unsigned s;
    const unsigned r = row_slot((unsigned)D.nx + 2u, &s), row = min(r, rows - 1u);
    const int p = (int)s - 1, k = (int)(row / (unsigned)D.ny), j = (int)(row - (unsigned)k * (unsigned)D.ny);
    const int ijk[3] = {0, j, k};
    bool store = r < rows && p >= 0 && p < D.nx && mid_lane();
    if (near_line(D, 0, ijk)) store = store && !near_pos(near_range(D, 0, D.nx), p, D.nx);
    row_unit<T, false>(D, store, p, j, k);
}
template <typename T>
__global__ void __launch_bounds__(128, 3) k3_near_row(Desc D, Near N) {
    const unsigned rows = (unsigned)(D.rn[1] * D.rn[2]);
    unsigned s;
    const unsigned r = row_slot((unsigned)N.len + 2u, &s), row = min(r, rows - 1u);
    const int k = D.r0[2] + (int)(row / (unsigned)D.rn[1]), j = D.r0[1] + (int)(row % (unsigned)D.rn[1]);
    const bool store = r < rows && s >= 1u && s <= (unsigned)N.len && mid_lane();
    int p = N.a + (int)s - 1;
    if (D.bc[0] == MB_BC_PERIODIC) {   // a cell's own position (its neighbours' are mapped)
        p %= D.nx;
        if (p < 0) p += D.nx;
    }
    row_unit<T, true>(D, store, p, j, k);
}

// y and z sweeps: a thread marches along seg cells of its line with a
// register window, 32 neighbouring lines per warp (along x, running on over
// the row's end), so that loads and stores are whole rows
template <typename T, int d, bool GEN>
__device__ __forceinline__ void march(const Desc &D, bool in, bool nearl, const int *line, int base, int stride,
                                      int m0, int m1, int nal) {
    using S = typename Flow<T, d>::S;
    const Flow<T, d> fl(D);
    const T *__restrict__ Q = qsrc<T>(D) + base;
    auto load = [&](int m, T *q, bool &fu) {
        bool flip;
        const int p = line_pos(D, d, m, nal, &flip);
        for (int k = 0; k < NC; ++k) q[k] = Q[(size_t)k * D.n + (size_t)p * stride];
        if (flip) q[1 + d] = -q[1 + d];
        fu = true;
        if (GEN) {
            int ijk[3] = {line[0], line[1], line[2]};
            ijk[d] = p;
            fu = fluid_a(D, ijk[0], ijk[1], ijk[2]);
        }
    };
    const Near N = near_range(D, d, nal);
    T qm[NC], qc[NC], qp[NC], qq[NC];
    bool um, uc, up, uq;
    S L, R, Rc;
    FluxT<T, GEN> F[NC], Fp[NC];
    double w[NC] = {0, 0, 0, 0, 0};
    {
        T qa[NC];
        bool ua;
        load(m0 - 2, qa, ua);
        load(m0 - 1, qm, um);
        load(m0, qc, uc);
        load(m0 + 1, qp, up);
        fl.states(qa, qm, qc, ua && uc, L, Rc);
    }
    for (int f = m0; f <= m1; ++f) {
        if (f < m1) load(f + 2, qq, uq);   // the next face's high neighbour
        double Qd[NC];
        const int c = base + (f - 1) * stride;
        const bool store = f > m0 && in && (GEN || !(nearl && near_pos(N, f - 1, nal)));
        if (sizeof(T) == 4) {
            if (store)
                for (int k = 0; k < NC; ++k) Qd[k] = D.Q[(size_t)k * D.n + c];
        } else {
            for (int k = 0; k < NC; ++k) Qd[k] = qm[k];
        }
        fl.states(qm, qc, qp, um && up, L, R);
        line_flux<T, d, GEN>(D, fl, line, f, nal, um && uc, Rc, L, F);
        if (store) line_update<T, d, GEN>(D, line, f - 1, nal, c, Qd, Fp, F, w);
        Rc = R;
        um = uc; uc = up; up = uq;
        for (int k = 0; k < NC; ++k) {
            Fp[k] = F[k];
            qm[k] = qc[k];
            qc[k] = qp[k];
            qp[k] = qq[k];
        }
    }
    if (GEN) add_wall(D, w);
}
template <typename T, int d>
__global__ void __launch_bounds__(32, 12) k3_march(Desc D, int seg, unsigned nlb) {
    const unsigned sg = blockIdx.x / nlb, lb = blockIdx.x - sg * nlb;
    const int nal = d == 1 ? D.ny : D.nz, nlines = D.n / nal;
    const int l = (int)(lb * 32u + threadIdx.x);
    const bool in = l < nlines;
    const int lc = in ? l : nlines - 1;
    const int i = lc % D.nx, o = lc / D.nx;   // o: the line's other coordinate (z for d = 1, y for d = 2)
    const int line[3] = {i, d == 1 ? 0 : o, d == 1 ? o : 0};
    const int m0 = (int)sg * seg, m1 = min(nal, m0 + seg);
    const int base = d == 1 ? o * D.ny * D.nx + i : lc, stride = d == 1 ? D.nx : D.nx * D.ny;
    march<T, d, false>(D, in, near_line(D, d, line), line, base, stride, m0, m1, nal);
}
// the near cells of a y or z sweep, one per thread
template <typename T, int d>
__global__ void __launch_bounds__(128, 3) k3_near(Desc D, Near N) {
    const int nal = d == 1 ? D.ny : D.nz, no = d == 1 ? D.rn[2] : D.rn[1];
    const int t = (int)(blockIdx.x * 128u + threadIdx.x), tot = D.rn[0] * no * N.len;
    const bool in = t < tot;
    const int tc = in ? t : tot - 1;
    const int i = D.r0[0] + tc % D.rn[0], o = D.r0[d == 1 ? 2 : 1] + (tc / D.rn[0]) % no;
    int m = N.a + tc / (D.rn[0] * no);
    if (D.bc[2 * d] == MB_BC_PERIODIC) {
        m %= nal;
        if (m < 0) m += nal;
    }
    const int line[3] = {i, d == 1 ? 0 : o, d == 1 ? o : 0};
    const int base = d == 1 ? o * D.ny * D.nx + i : o * D.nx + i, stride = d == 1 ? D.nx : D.nx * D.ny;
    march<T, d, true>(D, in, true, line, base, stride, m, m + 1, nal);
}

// covering / uncovering (Sec. II.C.5): each event cell of R finds its
// neighbour set, the face neighbours, else those sharing an edge, else a
// vertex (recipients: alpha_B > 0, and in donor mode alpha_A > 0), and the
// sum of their alpha_B
__global__ void k3_evprep(Desc D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= D.rn[0] * D.rn[1] * D.rn[2]) return;
    int i, j, k;
    r_cell(D, t, &i, &j, &k);
    const double aA = D.aA[t], aB = D.aB[t];
    const bool covered = aA > 0.0 && aB == 0.0;
    const bool unc = !D.gcl && aA == 0.0 && aB > 0.0;
    D.evt[t] = 0;
    if (!covered && !unc) return;
    unsigned mask = 0u;
    double asum = 0.0;
    for (int pass = 0; pass < 3 && mask == 0u; ++pass)
        for (int dk = -1; dk <= 1; ++dk)
            for (int dj = -1; dj <= 1; ++dj)
                for (int di = -1; di <= 1; ++di) {
                    const int nzc = (di != 0) + (dj != 0) + (dk != 0);
                    if (nzc == 0 || nzc > pass + 1) continue;
                    int ii, jj, kk;
                    if (nbr(D, i, j, k, di, dj, dk, &ii, &jj, &kk) < 0) continue;
                    const double b = alphaB(D, ii, jj, kk);
                    if (!(b > 0.0)) continue;
                    if (!D.gcl && alphaA(D, ii, jj, kk) == 0.0) continue;
                    mask |= 1u << ((dk + 1) * 9 + (dj + 1) * 3 + (di + 1));
                    asum += b;
                }
    if (mask == 0u) {
        const bool open = (D.bc[0] == MB_BC_TRANSMISSIVE && i == 0) || (D.bc[1] == MB_BC_TRANSMISSIVE && i == D.nx - 1) ||
                          (D.bc[2] == MB_BC_TRANSMISSIVE && j == 0) || (D.bc[3] == MB_BC_TRANSMISSIVE && j == D.ny - 1) ||
                          (D.bc[4] == MB_BC_TRANSMISSIVE && k == 0) || (D.bc[5] == MB_BC_TRANSMISSIVE && k == D.nz - 1);
        if (covered && open) D.evt[t] = 3;
        else atomicOr(D.err, E_NONBR);
        return;
    }
    D.evt[t] = covered ? 1 : 2;
    D.emask[t] = mask;
    D.easum[t] = asum;
}

// the events applied simultaneously, each cell of R gathering the changes
// to its own content in increasing order of the event cells (the order of
// the one-pass definition)
__global__ void k3_events(Desc D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= D.rn[0] * D.rn[1] * D.rn[2]) return;
    int i, j, k;
    r_cell(D, t, &i, &j, &k);
    const int c = cidx(D, i, j, k);
    const unsigned char e = D.evt[t];
    if (e == 1 || e == 3) {   // covered: its content leaves it
        for (int q = 0; q < NC; ++q) D.Cn[(size_t)q * D.n + c] = 0.0;
        return;
    }
    if (e == 2) {             // uncovered (donor mode): sigma times its donors' contents
        const double sigma = D.aB[t] / (D.aB[t] + D.easum[t]);
        const unsigned mask = D.emask[t];
        for (int q = 0; q < NC; ++q) {
            double tot = 0.0;
            for (int o = 0; o < 27; ++o) {
                if (!((mask >> o) & 1u)) continue;
                int ii, jj, kk;
                const int cc = nbr(D, i, j, k, o % 3 - 1, (o / 3) % 3 - 1, o / 9 - 1, &ii, &jj, &kk);
                tot += D.C[(size_t)q * D.n + cc];
            }
            D.Cn[(size_t)q * D.n + c] = sigma * tot;
        }
        D.upd[t] = 1;
        return;
    }
    // a recipient or donor: the event cells among the 26 neighbours that
    // name this cell, in increasing cell index
    int ev[26], ecell[26], ne = 0;
    for (int o = 0; o < 27; ++o) {
        if (o == 13) continue;
        int ii, jj, kk;
        const int cc = nbr(D, i, j, k, o % 3 - 1, (o / 3) % 3 - 1, o / 9 - 1, &ii, &jj, &kk);
        if (cc < 0 || !in_r(D, ii, jj, kk)) continue;
        const int r = ridx(D, ii, jj, kk);
        const unsigned char et = D.evt[r];
        if (et != 1 && et != 2) continue;
        // this cell seen from the event cell: the opposite offset
        const int ob = 26 - o;
        if (!((D.emask[r] >> ob) & 1u)) continue;
        int z = ne++;
        while (z > 0 && ecell[z - 1] > cc) { ecell[z] = ecell[z - 1]; ev[z] = ev[z - 1]; --z; }
        ecell[z] = cc;
        ev[z] = r;
    }
    if (ne == 0) return;
    const double aBc = alphaB(D, i, j, k);
    for (int q = 0; q < NC; ++q) {
        double x = D.Cn[(size_t)q * D.n + c];
        for (int m = 0; m < ne; ++m) {
            const int r = ev[m];
            if (D.evt[r] == 1) x += aBc / D.easum[r] * D.C[(size_t)q * D.n + ecell[m]];
            else x -= D.aB[r] / (D.aB[r] + D.easum[r]) * D.C[(size_t)q * D.n + c];
        }
        D.Cn[(size_t)q * D.n + c] = x;
    }
}

// safeguard seeds: non-physical new contents, and cells keeping less than
// COLLAPSE of their volume over the sweep, in the list (cell indices)
// (cells outside R are tested by the line kernels, whose contents no later step
// before the safeguard changes; this kernel runs over R, after the events)
__global__ void k3_bad(Desc D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= D.rn[0] * D.rn[1] * D.rn[2]) return;
    int i, j, k;
    r_cell(D, t, &i, &j, &k);
    const int c = cidx(D, i, j, k);
    if (!D.upd[t]) return;
    const double aB = D.aB[t];
    if (!(aB > 0.0)) return;
    double q[NC];
    for (int m = 0; m < NC; ++m) q[m] = D.Cn[(size_t)m * D.n + c];
    if (content_bad(q) || aB < COLLAPSE * D.aA[t]) add_seed(D, c);
}

// the merges (one thread): each cluster of seeds and their fluid, updated
// face neighbours shares its content in proportion to alpha_B; sums in cell
// order; cells still non-physical seed the next merge
__device__ bool physical5(const Desc &D, int c) {
    const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
    const double aB = alphaB(D, i, j, k);
    double q[NC];
    for (int m = 0; m < NC; ++m) {
        q[m] = D.Cn[(size_t)m * D.n + c] / aB;
        if (!isfinite(q[m])) return false;
    }
    return q[0] > 0.0 && pressure5(D.gamma, q) > 0.0;
}
// a merged cell's content; its FP32 copy too (in R k3_final writes it again)
__device__ __forceinline__ void put_share(const Desc &D, int c, int q, double v) {
    D.Cn[(size_t)q * D.n + c] = v;
    if (D.f32) D.Qfn[(size_t)q * D.n + c] = float(v);
}
// (one thread, over global lists: the form for clusters too large for the
// shared-memory form in k3_mix; it continues from layer layer0 with the ns
// seeds in D.seeds and the mixed count so far)
__device__ void mix_serial(const Desc &D, int ns, int layer0, int mixed) {
    int *seed = D.seeds;
    for (int layer = layer0; layer < MIX_LAYERS && ns > 0; ++layer) {
        // seeds in cell order
        for (int x = 1; x < ns; ++x) {
            const int v = seed[x];
            int z = x;
            while (z > 0 && seed[z - 1] > v) { seed[z] = seed[z - 1]; --z; }
            seed[z] = v;
        }
        int nn = 0;
        bool over = false;
        auto add = [&](int c) -> int {
            if (D.lab[c] >= 0) return D.lab[c];
            if (nn >= NODECAP) { over = true; return -1; }
            D.lab[c] = nn;
            D.nodes[nn] = c;
            D.par_[nn] = nn;
            return nn++;
        };
        auto root = [&](int a) { while (D.par_[a] != a) a = D.par_[a]; return a; };
        for (int s = 0; s < ns && !over; ++s) {
            const int c = seed[s];
            const int a = add(c);
            if (a < 0) break;
            const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
            const int off[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
            for (int m = 0; m < 6; ++m) {
                int ii, jj, kk;
                const int cc = nbr(D, i, j, k, off[m][0], off[m][1], off[m][2], &ii, &jj, &kk);
                if (cc < 0 || !(alphaB(D, ii, jj, kk) > 0.0) || !updated(D, ii, jj, kk)) continue;
                const int b = add(cc);
                if (b < 0) break;
                const int ra = root(a), rb = root(b);
                // the root is the smaller cell index
                if (ra != rb) { if (D.nodes[ra] < D.nodes[rb]) D.par_[rb] = ra; else D.par_[ra] = rb; }
            }
        }
        if (over) {
            *D.err |= E_NODECAP;
            for (int m = 0; m < nn; ++m) D.lab[D.nodes[m]] = -1;
            return;
        }
        // every node's root cell (by insertion index), then the nodes in
        // cell order with their root cells
        int *rootcell = D.seeds + SEEDCAP;     // scratch after the seeds
        for (int x = 0; x < nn; ++x) rootcell[x] = D.nodes[root(x)];
        for (int x = 1; x < nn; ++x) {
            const int v = D.nodes[x], rv = rootcell[x];
            int z = x;
            while (z > 0 && D.nodes[z - 1] > v) { D.nodes[z] = D.nodes[z - 1]; rootcell[z] = rootcell[z - 1]; --z; }
            D.nodes[z] = v;
            rootcell[z] = rv;
        }
        // each cluster's sums at the slot of its root cell (its position
        // among the sorted nodes), members added in cell order
        for (int x = 0; x < nn; ++x) for (int q = 0; q <= NC; ++q) D.ntot[(NC + 1) * x + q] = 0.0;
        auto slot = [&](int cell) {
            int lo = 0, hi = nn - 1;
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (D.nodes[mid] < cell) lo = mid + 1; else hi = mid; }
            return lo;
        };
        for (int x = 0; x < nn; ++x) {
            const int c = D.nodes[x];
            const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
            const int sr = slot(rootcell[x]);
            D.ntot[(NC + 1) * sr + NC] += alphaB(D, i, j, k);
            for (int q = 0; q < NC; ++q) D.ntot[(NC + 1) * sr + q] += D.Cn[(size_t)q * D.n + c];
        }
        for (int x = 0; x < nn; ++x) {
            const int c = D.nodes[x];
            const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
            const int sr = slot(rootcell[x]);
            const double aB = alphaB(D, i, j, k);
            for (int q = 0; q < NC; ++q)
                put_share(D, c, q, aB * (D.ntot[(NC + 1) * sr + q] / D.ntot[(NC + 1) * sr + NC]));
        }
        mixed += nn;
        // cells still non-physical, in cell order
        int nb = 0;
        for (int x = 0; x < nn; ++x) {
            const int c = D.nodes[x];
            if (!physical5(D, c)) seed[nb++] = c;
        }
        for (int x = 0; x < nn; ++x) D.lab[D.nodes[x]] = -1;
        ns = nb;
    }
    if (ns > 0) atomicOr(D.err, E_UNSTABLE);   // cells left non-physical after the last merge
    *D.mixed = mixed;
}

// The merges in one 256-thread block over shared memory, while a layer's
// seeds and nodes fit (MIXS_SEEDS seeds, MIXS_NODES nodes); else the
// remaining layers in mix_serial.  The same clusters, sums and write-back
// as mix_serial: the candidate cells (the seeds and their fluid, updated
// face neighbours) are sorted and made unique (the nodes, in cell order);
// the clusters are the connected components of the seed-neighbour edges,
// labelled by their smallest node (repeated minimum over the edges until
// no label changes); each cluster's smallest node's thread sums its
// members in node order, i.e. in cell order.
constexpr int MIXS_THREADS = 256, MIXS_SORT = 1024, MIXS_SEEDS = MIXS_SORT / 7, MIXS_NODES = 320;
__device__ __forceinline__ int node_of(const int *nodes, int nn, int c) {
    int lo = 0, hi = nn - 1;
    while (lo < hi) { const int mid = (lo + hi) >> 1; if (nodes[mid] < c) lo = mid + 1; else hi = mid; }
    return lo;
}
__global__ void __launch_bounds__(MIXS_THREADS) k3_mix(Desc D) {
    __shared__ int cand[MIXS_SORT];
    __shared__ int enode[MIXS_SEEDS * 6];   // per (seed, direction): the neighbour's cell, then its node; -1 none
    __shared__ int snode[MIXS_SEEDS];       // the seed's node
    __shared__ int nodes[MIXS_NODES], lbl[MIXS_NODES];
    __shared__ double cache[MIXS_NODES][NC + 1], sums[MIXS_NODES][NC + 1];
    __shared__ int s_wsum[MIXS_THREADS / 32], s_changed, s_nb;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int ns = *D.nseed;
    if (ns > SEEDCAP) {
        if (tid == 0) atomicOr(D.err, E_SEEDCAP);
        ns = SEEDCAP;
    }
    int mixed = 0, layer = 0;
    for (; layer < MIX_LAYERS && ns > 0; ++layer) {
        if (ns > MIXS_SEEDS) break;
        int P = 2;
        while (P < 7 * ns) P <<= 1;
        // candidates: seed s at 7s, its neighbours after it
        for (int x = tid; x < P; x += MIXS_THREADS) cand[x] = INT_MAX;
        __syncthreads();
        for (int s = tid; s < ns; s += MIXS_THREADS) {
            const int c = D.seeds[s];
            const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
            cand[7 * s] = c;
            const int off[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
            for (int m = 0; m < 6; ++m) {
                int ii, jj, kk;
                const int cc = nbr(D, i, j, k, off[m][0], off[m][1], off[m][2], &ii, &jj, &kk);
                const bool ok = cc >= 0 && alphaB(D, ii, jj, kk) > 0.0 && updated(D, ii, jj, kk);
                cand[7 * s + 1 + m] = ok ? cc : INT_MAX;
                enode[6 * s + m] = ok ? cc : -1;
            }
        }
        __syncthreads();
        // bitonic sort of cand[0, P)
        for (int k2 = 2; k2 <= P; k2 <<= 1)
            for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
                for (int x = tid; x < P; x += MIXS_THREADS) {
                    const int y = x ^ j2;
                    if (y > x) {
                        const int a = cand[x], b = cand[y];
                        if ((a > b) == ((x & k2) == 0)) { cand[x] = b; cand[y] = a; }
                    }
                }
                __syncthreads();
            }
        // the distinct cells, in order: a contiguous chunk per thread and a
        // block-wide exclusive scan of the chunks' counts
        const int per = (P + MIXS_THREADS - 1) / MIXS_THREADS, x0 = min(P, tid * per), x1 = min(P, x0 + per);
        int cnt = 0;
        for (int x = x0; x < x1; ++x) cnt += cand[x] != INT_MAX && (x == 0 || cand[x - 1] != cand[x]);
        int inc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_wsum[wid] = inc;
        __syncthreads();
        int pos = inc - cnt, tot = 0;
        for (int w = 0; w < MIXS_THREADS / 32; ++w) {
            if (w < wid) pos += s_wsum[w];
            tot += s_wsum[w];
        }
        for (int x = x0; x < x1; ++x)
            if (cand[x] != INT_MAX && (x == 0 || cand[x - 1] != cand[x])) {
                if (pos < MIXS_NODES) nodes[pos] = cand[x];
                ++pos;
            }
        __syncthreads();
        const int nn = tot;
        if (nn > MIXS_NODES) break;
        // edges as node pairs, labels, the nodes' contents and alpha_B
        for (int x = tid; x < 6 * ns; x += MIXS_THREADS)
            if (enode[x] >= 0) enode[x] = node_of(nodes, nn, enode[x]);
        for (int s = tid; s < ns; s += MIXS_THREADS) snode[s] = node_of(nodes, nn, D.seeds[s]);
        for (int x = tid; x < nn; x += MIXS_THREADS) {
            const int c = nodes[x];
            const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
            lbl[x] = x;
            for (int q = 0; q < NC; ++q) cache[x][q] = D.Cn[(size_t)q * D.n + c];
            cache[x][NC] = alphaB(D, i, j, k);
        }
        for (;;) {
            __syncthreads();
            if (tid == 0) s_changed = 0;
            __syncthreads();
            for (int x = tid; x < 6 * ns; x += MIXS_THREADS) {
                const int b = enode[x];
                if (b < 0) continue;
                const int a = snode[x / 6];
                const int la = lbl[a], lb = lbl[b];
                if (la != lb) {
                    const int mn = min(la, lb);
                    atomicMin(&lbl[a], mn);
                    atomicMin(&lbl[b], mn);
                    s_changed = 1;
                }
            }
            __syncthreads();
            const int ch = s_changed;
            if (!ch) break;
        }
        // each cluster's sums (alpha_B and contents) in node order
        for (int r = tid; r < nn; r += MIXS_THREADS) {
            if (lbl[r] != r) continue;
            double acc[NC + 1] = {0, 0, 0, 0, 0, 0};
            for (int x = r; x < nn; ++x) {
                if (lbl[x] != r) continue;
                acc[NC] += cache[x][NC];
                for (int q = 0; q < NC; ++q) acc[q] += cache[x][q];
            }
            for (int q = 0; q <= NC; ++q) sums[r][q] = acc[q];
        }
        if (tid == 0) s_nb = 0;
        __syncthreads();
        // shares in proportion to alpha_B; cells still non-physical seed
        // the next layer (its candidates are sorted, so order is free)
        for (int x = tid; x < nn; x += MIXS_THREADS) {
            const int c = nodes[x], r = lbl[x];
            const double aB = cache[x][NC];
            for (int q = 0; q < NC; ++q) put_share(D, c, q, aB * (sums[r][q] / sums[r][NC]));
            if (!physical5(D, c)) D.seeds[atomicAdd(&s_nb, 1)] = c;
        }
        mixed += nn;
        __syncthreads();
        ns = s_nb;
        __syncthreads();
    }
    if (layer < MIX_LAYERS && ns > 0) {   // too large for shared memory: the serial form goes on
        if (tid == 0) mix_serial(D, ns, layer, mixed);
        return;
    }
    if (tid == 0 && ns > 0) atomicOr(D.err, E_UNSTABLE);   // cells left non-physical after the last merge
    if (tid == 0) *D.mixed = mixed;
}

// Q = content / alpha_B (NaN where alpha_B = 0 or the cell was not
// updated) in R, in place, with the checks of the new state.  Elsewhere
// alpha_B = 1 and the content is the state: its test was the seed test, and
// the safeguard flags cells it leaves non-physical.
__global__ void k3_final(Desc D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= D.rn[0] * D.rn[1] * D.rn[2]) return;
    int i, j, k;
    r_cell(D, t, &i, &j, &k);
    const int c = cidx(D, i, j, k);
    const double aB = D.aB[t];
    const bool ok = aB > 0.0 && D.upd[t];
    const double ia = ok ? (aB == 1.0 ? 1.0 : 1.0 / aB) : 0.0;
    double q[NC];
    for (int m = 0; m < NC; ++m) {
        const double cn = D.Cn[(size_t)m * D.n + c];
        q[m] = ok ? (ia == 1.0 ? cn : cn * ia) : NAN;
        D.Cn[(size_t)m * D.n + c] = q[m];
        if (D.f32) D.Qfn[(size_t)m * D.n + c] = float(q[m]);
        // the provisional state of a cell that was solid at pose A (k3_wall)
        // leaves the step-start state
        if (D.gcl && D.aA[t] == 0.0) D.Q[(size_t)m * D.n + c] = NAN;
    }
    if (aB > 0.0 && !D.upd[t]) atomicOr(D.err, E_UNSTABLE);
    if (ok) {
        bool bad = !(q[0] > 0.0) || !(2.0 * q[0] * q[4] > q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
        for (int m = 0; m < NC; ++m) if (!finite64(q[m])) bad = true;
        if (bad) atomicOr(D.err, E_UNSTABLE);
    }
}

// maxima of |u_d| + c over the fluid cells (positive doubles compare as
// their bit patterns), in the type T of the flow arithmetic; 256-thread
// blocks, one atomic per block and axis.
// FP64: a block takes 2048 cells at a time and first forms their speeds in
// FP32; only a cell within 1e-5 of the largest the block has seen along an
// axis, or one whose FP32 speeds are not trusted (speeds32), goes through the
// FP64 formula, so that the result is that formula's over every cell.  4 M cells: 267 us with the FP64 formula
// throughout.
constexpr int SPEED_CELLS = 8;   // cells per thread and turn (FP64)
template <typename T>
__device__ __forceinline__ void block_max3(const T *s, T (*red)[8], T *m) {
    for (int a = 0; a < 3; ++a) {
        T v = s[a];
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((threadIdx.x & 31) == 0) red[a][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    for (int a = 0; a < 3; ++a) {
        m[a] = red[a][0];
        for (int q = 1; q < 8; ++q) m[a] = fmax(m[a], red[a][q]);
    }
    __syncthreads();
}
__device__ __forceinline__ void put_speeds(const Desc &D, const double *v) {
    const int a = threadIdx.x;
    if (a < 3 && v[a] > 0.0)
        atomicMax((unsigned long long *)&D.smax[a], (unsigned long long)__double_as_longlong(v[a]));
}
__global__ void __launch_bounds__(256) k3_speeds64(Desc D) {
    __shared__ float redf[3][8];
    __shared__ double red[3][8];
    const double g = D.gamma;
    const float gf = D.gammaf, h1f = (float)D.g1h;
    double s[3] = {0.0, 0.0, 0.0};
    float lead[3] = {0.0f, 0.0f, 0.0f};
    for (long long c0 = (long long)blockIdx.x * 256 * SPEED_CELLS; c0 < D.n; c0 += (long long)gridDim.x * 256 * SPEED_CELLS) {
        float v[SPEED_CELLS][3], m[3] = {0.0f, 0.0f, 0.0f};
        unsigned want = 0u;
#pragma unroll
        for (int u = 0; u < SPEED_CELLS; ++u) {
            const long long c = c0 + u * 256 + threadIdx.x;
            v[u][0] = v[u][1] = v[u][2] = -1.0f;
            if (c >= D.n) continue;
            bool ok = true;
            float x[NC];
            bool fluid = true;
            for (int k = 0; k < NC; ++k) {
                const double q = D.Q[(size_t)k * D.n + c];
                if (k == 0) fluid = !isnan64(q);
                x[k] = near32(q, ok);
            }
            if (!fluid) continue;
            float ir, cs;
            if (!(speeds32<NC>(gf, h1f, x, ir, cs) && ok)) { want |= 1u << u; continue; }
            for (int a = 0; a < 3; ++a) {
                v[u][a] = fabsf(x[1 + a] * ir) + cs;
                m[a] = fmaxf(m[a], v[u][a]);
            }
        }
        float bm[3];
        block_max3<float>(m, redf, bm);
        for (int a = 0; a < 3; ++a) lead[a] = fmaxf(lead[a], bm[a]);
#pragma unroll
        for (int u = 0; u < SPEED_CELLS; ++u) {
            for (int a = 0; a < 3; ++a)
                if (v[u][a] >= lead[a] * (1.0f - 1e-5f)) want |= 1u << u;
        }
        while (want) {
            const int u = __ffs(want) - 1;
            want &= want - 1;
            const long long c = c0 + u * 256 + threadIdx.x;
            double q[NC];
            for (int k = 0; k < NC; ++k) q[k] = D.Q[(size_t)k * D.n + c];
            const double ir = rcp64(q[0]), p = press64<NC>(D.g1h, q, ir), cs = sqrt64(g * (p * ir));
            for (int a = 0; a < 3; ++a) {
                const double x = __fma_rn(abs64(q[1 + a]), ir, cs);
                if (pos64(x)) s[a] = max64(s[a], x);
            }
        }
    }
    double bm[3];
    block_max3<double>(s, red, bm);
    put_speeds(D, bm);
}
__global__ void __launch_bounds__(256) k3_speeds32(Desc D) {
    __shared__ float red[3][8];
    const float g = D.gammaf;
    float s[3] = {0.0f, 0.0f, 0.0f};
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < D.n; c += gridDim.x * blockDim.x) {
        float q[NC];
        for (int m = 0; m < NC; ++m) q[m] = D.Qf[(size_t)m * D.n + c];
        if (isnan(q[0])) continue;
        const float ir = 1.0f / q[0];
        const float p = (g - 1.0f) * (q[4] - 0.5f * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) * ir);
        const float cs = sqrtf(g * p * ir);
        for (int a = 0; a < 3; ++a) s[a] = fmaxf(s[a], fabsf(q[1 + a] * ir) + cs);
    }
    float bm[3];
    block_max3<float>(s, red, bm);
    const double v[3] = {(double)bm[0], (double)bm[1], (double)bm[2]};
    put_speeds(D, v);
}

// solid cells (alpha = 0 in R at the current pose) read NaN; alpha of every
// cell into out (optional)
__global__ void k3_classify(Desc D, double *alpha_out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= D.n) return;
    const int i = c % D.nx, j = (c / D.nx) % D.ny, k = c / (D.nx * D.ny);
    const double a = alphaA(D, i, j, k);
    if (alpha_out) alpha_out[c] = a;
    else if (!(a > 0.0)) for (int m = 0; m < NC; ++m) D.Q[(size_t)m * D.n + c] = NAN;
}

// the FP32 copy of the state (FP32 flux option)
__global__ void k3_to_f32(Desc D) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= D.n) return;
    for (int m = 0; m < NC; ++m) D.Qf[(size_t)m * D.n + c] = float(D.Q[(size_t)m * D.n + c]);
}

}  // namespace mb3

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
using mb3::Desc;
using mb3::NC;

struct mb3_sim {
    Desc D{};
    int nplane = 0;
    double pn[3 * MB3_MAX_PLANES] = {}, pc[MB3_MAX_PLANES] = {}, bb[6] = {};
    double t = 0.0, T[3] = {0.0, 0.0, 0.0};
    long step = 0;
    int sidx = 0;
    double dt_step = 0.0, cfl = 0.5;
    cudaStream_t st = nullptr;
    // the geometry (k3_cells, k3_faces, k3_swept side by side, then k3_wall)
    // beside the cells away from the body
    cudaStream_t gs[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t fork = nullptr, join[3] = {nullptr, nullptr, nullptr};
    std::string err;
    size_t rcap = 0, rfcap = 0;
    bool prev_ok = false;        // aB / tB hold the current pose over the region q0, qn
    int q0[3] = {0, 0, 0}, qn[3] = {0, 0, 0};
    // what a sweep reports (device: D.wall .. D.err in one block; host: one
    // page-locked slot per sweep of a step, filled without waiting)
    struct Report {
        double wall[NC];
        int mixed, nseed, err, pad;
    };
    Report *dev_report = nullptr, *report = nullptr;
    int last_report = 0;
    double *smax_host = nullptr;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};   // around the last sweep's two line launches
    float flux_ms = 0.0f;
    bool near_timed = false;
    std::vector<void *> owned;
};

static mb_status fail3(mb3_sim *s, mb_status r, const std::string &m) {
    if (s) s->err = m;
    return r;
}
static mb_status cuda3(mb3_sim *s, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return MB_OK;
    return fail3(s, e == cudaErrorMemoryAllocation ? MB_E_NOMEM : MB_E_CUDA,
                 std::string(what) + ": " + cudaGetErrorString(e));
}
template <class X>
static cudaError_t dalloc(mb3_sim *s, X **p, size_t count) {
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(1, count) * sizeof(X));
    if (e == cudaSuccess) s->owned.push_back(q);
    *p = (X *)q;
    return e;
}
static void dfree(mb3_sim *s, void *p) {
    if (!p) return;
    cudaFree(p);
    s->owned.erase(std::remove(s->owned.begin(), s->owned.end(), p), s->owned.end());
}

// the body posed at translation T
static mb3::Body3 posed(const mb3_sim *s, const double *T) {
    mb3::Body3 B;
    memset(&B, 0, sizeof(B));
    B.np = s->nplane;
    for (int f = 0; f < s->nplane; ++f) {
        for (int a = 0; a < 3; ++a) {
            B.n[3 * f + a] = s->pn[3 * f + a];
            B.nf[3 * f + a] = (float)s->pn[3 * f + a];
        }
        B.c[f] = s->pc[f] + (s->pn[3 * f] * T[0] + s->pn[3 * f + 1] * T[1] + s->pn[3 * f + 2] * T[2]);
        B.cf[f] = (float)B.c[f];
    }
    return B;
}

// region R: the cells meeting the body's bounding box at translations TA and
// TB, widened by two cells, inside the grid (rn = 0: no body in the grid)
static void region(mb3_sim *s, const double *TA, const double *TB, int *r0, int *rn) {
    const int nn[3] = {s->D.nx, s->D.ny, s->D.nz};
    for (int a = 0; a < 3; ++a) {
        r0[a] = 0;
        rn[a] = 0;
    }
    if (s->nplane == 0) return;
    for (int a = 0; a < 3; ++a) {
        const double u0 = std::min(s->bb[2 * a] + TA[a], s->bb[2 * a] + TB[a]);
        const double u1 = std::max(s->bb[2 * a + 1] + TA[a], s->bb[2 * a + 1] + TB[a]);
        long lo = (long)std::floor((u0 - s->D.lo[a]) / s->D.h[a]) - 2;
        long hi = (long)std::floor((u1 - s->D.lo[a]) / s->D.h[a]) + 2;
        lo = std::max(lo, 0L);
        hi = std::min(hi, (long)nn[a] - 1);
        if (hi < lo) { for (int q = 0; q < 3; ++q) rn[q] = 0; return; }
        r0[a] = (int)lo;
        rn[a] = (int)(hi - lo + 1);
    }
}

// R's buffers for at least rc cells and rf faces per axis
static cudaError_t ensure_r(mb3_sim *s, size_t rc, size_t rf) {
    cudaError_t e = cudaSuccess;
    Desc &D = s->D;
    if (rc > s->rcap) {
        cudaStreamSynchronize(s->st);
        dfree(s, D.aA); dfree(s, D.aM); dfree(s, D.aB); dfree(s, D.tA); dfree(s, D.tB); dfree(s, D.whas);
        dfree(s, D.aP); dfree(s, D.tP);
        s->prev_ok = false;
        dfree(s, D.wdist); dfree(s, D.wFB); dfree(s, D.wQB); dfree(s, D.evt); dfree(s, D.upd); dfree(s, D.emask); dfree(s, D.easum);
        const size_t c = rc + rc / 4;
        if (e == cudaSuccess) e = dalloc(s, &D.aA, c);
        if (e == cudaSuccess) e = dalloc(s, &D.aM, c);
        if (e == cudaSuccess) e = dalloc(s, &D.aB, c);
        if (e == cudaSuccess) e = dalloc(s, &D.tA, c);
        if (e == cudaSuccess) e = dalloc(s, &D.tB, c);
        if (e == cudaSuccess) e = dalloc(s, &D.aP, c);
        if (e == cudaSuccess) e = dalloc(s, &D.tP, c);
        if (e == cudaSuccess) e = dalloc(s, &D.whas, c);
        if (e == cudaSuccess) e = dalloc(s, &D.wdist, c);
        if (e == cudaSuccess) e = dalloc(s, &D.wFB, NC * c);
        if (e == cudaSuccess) e = dalloc(s, &D.wQB, NC * c);
        if (e == cudaSuccess) e = dalloc(s, &D.evt, c);
        if (e == cudaSuccess) e = dalloc(s, &D.upd, c);
        if (e == cudaSuccess) e = dalloc(s, &D.emask, c);
        if (e == cudaSuccess) e = dalloc(s, &D.easum, c);
        s->rcap = e == cudaSuccess ? c : 0;
    }
    if (e == cudaSuccess && rf > s->rfcap) {
        cudaStreamSynchronize(s->st);
        for (int a = 0; a < 3; ++a) dfree(s, D.bM[a]);
        dfree(s, D.bt);
        const size_t c = rf + rf / 4;
        for (int a = 0; a < 3 && e == cudaSuccess; ++a) e = dalloc(s, &D.bM[a], c);
        if (e == cudaSuccess) e = dalloc(s, &D.bt, c);
        s->rfcap = e == cudaSuccess ? c : 0;
    }
    return e;
}

static unsigned nblk(long long n, int b = 256) { return (unsigned)std::max<long long>(1, (n + b - 1) / b); }

// alpha at translation T over R(T) (into D.aA) and the classification
static cudaError_t pose_alpha(mb3_sim *s, const double *T, Desc &D) {
    region(s, T, T, D.r0, D.rn);
    const size_t rc = (size_t)D.rn[0] * D.rn[1] * D.rn[2];
    const size_t rf = (size_t)(D.rn[0] + 1) * (D.rn[1] + 1) * (D.rn[2] + 1);
    cudaError_t e = ensure_r(s, rc, rf);
    if (e != cudaSuccess) return e;
    D = s->D, region(s, T, T, D.r0, D.rn);
    if (rc > 0) {
        const mb3::Body3 B = posed(s, T);
        mb3::k3_cells<<<nblk(32LL * (long long)rc), 256, 0, s->st>>>(D, B, B, B, mb3::CELLS_ONE);   // one pose
    }
    e = cudaGetLastError();
    s->prev_ok = e == cudaSuccess;
    for (int a = 0; a < 3; ++a) { s->q0[a] = D.r0[a]; s->qn[a] = D.rn[a]; }
    return e;
}

extern "C" {

mb_status mb3_create(const mb3_grid *g, double gamma, double cfl, const mb3_body *b, int uncover_mode,
                     mb3_sim **out) {
    if (!out) return MB_E_INVAL;
    *out = nullptr;
    if (!g || !b) return MB_E_INVAL;
    if (g->nx < 1 || g->ny < 1 || g->nz < 1 || (long long)g->nx * g->ny * g->nz > (1LL << 30)) return MB_E_INVAL;
    for (int a = 0; a < 3; ++a) if (!(g->hi[a] > g->lo[a])) return MB_E_INVAL;
    for (int q = 0; q < 6; ++q) if (g->bc[q] < 0 || g->bc[q] > 2) return MB_E_INVAL;
    for (int a = 0; a < 3; ++a) if ((g->bc[2 * a] == MB_BC_PERIODIC) != (g->bc[2 * a + 1] == MB_BC_PERIODIC)) return MB_E_INVAL;
    // the stencil's two ghost cells mirror two cells of a non-periodic axis
    const int nax[3] = {g->nx, g->ny, g->nz};
    for (int a = 0; a < 3; ++a) if (nax[a] < 2 && g->bc[2 * a] != MB_BC_PERIODIC) return MB_E_INVAL;
    if (!(gamma > 1.0) || !(cfl > 0.0 && cfl <= 1.0)) return MB_E_INVAL;
    if (uncover_mode != MB_UNCOVER_DONOR && uncover_mode != MB_UNCOVER_FLUX_GCL) return MB_E_INVAL;
    if (b->nplane < 0 || b->nplane > MB3_MAX_PLANES || (b->nplane > 0 && (!b->normals || !b->offsets))) return MB_E_INVAL;
    mb3_sim *s = new mb3_sim();
    Desc &D = s->D;
    D.nx = g->nx; D.ny = g->ny; D.nz = g->nz;
    D.n = g->nx * g->ny * g->nz;
    const int nn[3] = {g->nx, g->ny, g->nz};
    for (int a = 0; a < 3; ++a) {
        D.lo[a] = g->lo[a];
        D.h[a] = (g->hi[a] - g->lo[a]) / nn[a];
        D.lof[a] = (float)D.lo[a];
        D.hf[a] = (float)D.h[a];
        D.bigf[a] = (float)(std::fabs(g->lo[a]) + (g->hi[a] - g->lo[a]) + 2.0 * D.h[a]);
        D.U[a] = b->U[a];
    }
    for (int q = 0; q < 6; ++q) D.bc[q] = g->bc[q];
    D.gamma = gamma;
    D.g1h = 0.5 * (gamma - 1.0);
    D.gammaf = (float)gamma;
    D.gcl = uncover_mode == MB_UNCOVER_FLUX_GCL;
    s->cfl = cfl;
    s->nplane = b->nplane;
    for (int f = 0; f < b->nplane; ++f) {
        for (int a = 0; a < 3; ++a) s->pn[3 * f + a] = b->normals[3 * f + a];
        s->pc[f] = b->offsets[f];
    }
    for (int q = 0; q < 6; ++q) s->bb[q] = b->bbox[q];
    cudaError_t e = cudaStreamCreateWithFlags(&s->st, cudaStreamNonBlocking);
    for (int q = 0; q < 4 && e == cudaSuccess; ++q) e = cudaEventCreate(&s->ev[q]);
    int plo = 0, phi = 0;
    if (e == cudaSuccess) e = cudaDeviceGetStreamPriorityRange(&plo, &phi);
    for (int q = 0; q < 3 && e == cudaSuccess; ++q) {
        e = cudaStreamCreateWithPriority(&s->gs[q], cudaStreamNonBlocking, phi);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->join[q], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->fork, cudaEventDisableTiming);
    const size_t n = D.n;
    if (e == cudaSuccess) e = dalloc(s, &D.Q, NC * n);
    if (e == cudaSuccess) e = dalloc(s, &D.Qn, NC * n);
    if (e == cudaSuccess) e = dalloc(s, &D.C, NC * n);
    if (e == cudaSuccess) e = dalloc(s, &D.Cn, NC * n);
    if (e == cudaSuccess) e = dalloc(s, &s->dev_report, 1);
    if (e == cudaSuccess) {
        D.wall = s->dev_report->wall;
        D.mixed = &s->dev_report->mixed;
        D.nseed = &s->dev_report->nseed;
        D.err = &s->dev_report->err;
        e = cudaHostAlloc((void **)&s->report, 3 * sizeof(mb3_sim::Report) + 3 * sizeof(double), cudaHostAllocDefault);
    }
    if (e == cudaSuccess) {
        memset(s->report, 0, 3 * sizeof(mb3_sim::Report));
        s->smax_host = (double *)(s->report + 3);
    }
    if (e == cudaSuccess) e = dalloc(s, &D.seeds, mb3::SEEDCAP + mb3::NODECAP);
    if (e == cudaSuccess) e = dalloc(s, &D.lab, n);
    if (e == cudaSuccess) e = dalloc(s, &D.par_, mb3::NODECAP);
    if (e == cudaSuccess) e = dalloc(s, &D.nodes, mb3::NODECAP);
    if (e == cudaSuccess) e = dalloc(s, &D.ntot, (NC + 1) * (size_t)mb3::NODECAP);
    if (e == cudaSuccess) e = dalloc(s, &D.smax, 3);
    if (e == cudaSuccess) e = cudaMemsetAsync(D.lab, 0xff, n * sizeof(int), s->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(D.err, 0, sizeof(int), s->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(D.Q, 0, NC * n * sizeof(double), s->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) {
        const mb_status r = e == cudaErrorMemoryAllocation ? MB_E_NOMEM : MB_E_CUDA;
        mb3_destroy(s);
        return r;
    }
    *out = s;
    return MB_OK;
}

void mb3_destroy(mb3_sim *s) {
    if (!s) return;
    if (s->st) cudaStreamSynchronize(s->st);
    for (int q = 0; q < 3; ++q) if (s->gs[q]) cudaStreamSynchronize(s->gs[q]);
    for (void *p : s->owned) cudaFree(p);
    if (s->report) cudaFreeHost(s->report);
    for (int q = 0; q < 4; ++q) if (s->ev[q]) cudaEventDestroy(s->ev[q]);
    if (s->fork) cudaEventDestroy(s->fork);
    for (int q = 0; q < 3; ++q) {
        if (s->join[q]) cudaEventDestroy(s->join[q]);
        if (s->gs[q]) cudaStreamDestroy(s->gs[q]);
    }
    if (s->st) cudaStreamDestroy(s->st);
    delete s;
}

const char *mb3_last_error(const mb3_sim *s) { return s ? s->err.c_str() : "NULL simulation"; }

static mb_status err_status(mb3_sim *s, int w) {
    if (w & (mb3::E_SEEDCAP | mb3::E_NODECAP))
        return fail3(s, MB_E_CAPACITY, "positivity safeguard: more cells than its lists hold");
    if (w & mb3::E_NONBR) return fail3(s, MB_E_UNSTABLE, "covered/uncovered cell without a fluid neighbour");
    if (w & mb3::E_UNSTABLE) return fail3(s, MB_E_UNSTABLE, "non-physical state after the safeguard");
    return MB_OK;
}

mb_status mb3_write_state(mb3_sim *s, const double *Q, double t, const double *T) {
    if (!s || !Q || !T) return MB_E_INVAL;
    cudaError_t e = cudaMemcpyAsync(s->D.Q, Q, NC * (size_t)s->D.n * sizeof(double), cudaMemcpyHostToDevice, s->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->D.err, 0, sizeof(int), s->st);
    Desc D = s->D;
    if (e == cudaSuccess) e = pose_alpha(s, T, D);
    if (e == cudaSuccess) mb3::k3_classify<<<nblk(s->D.n), 256, 0, s->st>>>(D, nullptr);
    if (e == cudaSuccess && D.f32) mb3::k3_to_f32<<<nblk(s->D.n), 256, 0, s->st>>>(D);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_write_state");
    s->t = t;
    for (int a = 0; a < 3; ++a) s->T[a] = T[a];
    s->step = 0;
    s->sidx = 0;
    return MB_OK;
}

mb_status mb3_read_state(mb3_sim *s, double *Q, double *alpha, double *clock) {
    if (!s) return MB_E_INVAL;
    cudaError_t e = cudaSuccess;
    if (Q) e = cudaMemcpyAsync(Q, s->D.Q, NC * (size_t)s->D.n * sizeof(double), cudaMemcpyDeviceToHost, s->st);
    if (alpha && e == cudaSuccess) {
        Desc D = s->D;
        e = pose_alpha(s, s->T, D);
        if (e == cudaSuccess) mb3::k3_classify<<<nblk(s->D.n), 256, 0, s->st>>>(D, s->D.C);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(alpha, s->D.C, (size_t)s->D.n * sizeof(double), cudaMemcpyDeviceToHost, s->st);
    }
    int w = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&w, s->D.err, sizeof(int), cudaMemcpyDeviceToHost, s->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_read_state");
    if (clock) {
        clock[0] = s->t;
        for (int a = 0; a < 3; ++a) clock[1 + a] = s->T[a];
        clock[4] = (double)s->step;
    }
    return err_status(s, w);
}

// the line kernels of a sweep along D.d: over all but the near cells, or over
// those (near)
extern "C++" {
template <typename T>
static void line_sweep_t(const Desc &D, bool near, cudaStream_t st) {
    const int nal = D.d == 0 ? D.nx : D.d == 1 ? D.ny : D.nz;
    if (near) {
        const mb3::Near N = mb3::near_range(D, D.d, nal);
        if (N.len == 0) return;
        const long long cells = (long long)N.len * D.rn[0] * D.rn[1] * D.rn[2] / D.rn[D.d];
        const long long slots = (long long)(N.len + 2) * D.rn[1] * D.rn[2];
        if (D.d == 0) mb3::k3_near_row<T><<<nblk((slots + 29) / 30 * 32, 128), 128, 0, st>>>(D, N);
        else if (D.d == 1) mb3::k3_near<T, 1><<<nblk(cells, 128), 128, 0, st>>>(D, N);
        else mb3::k3_near<T, 2><<<nblk(cells, 128), 128, 0, st>>>(D, N);
        return;
    }
    if (D.d == 0) {
        const long long slots = (long long)(D.nx + 2) * D.ny * D.nz;
        mb3::k3_row<T><<<nblk((slots + 29) / 30 * 32, 128), 128, 0, st>>>(D);
        return;
    }
    // cells per thread: a segment costs two evolved states and a flux more
    // than its cells, so as long as leaves 32 warps per SM (8 per quarter,
    // each with its share of the FP64 pipe), from 64 down to 8, in CTAs of one
    // warp.  200 x 200 x 100 cells, FP64: 1.51 ms with 16 warps per SM
    const unsigned nlb = nblk(D.n / nal, 32);
    int seg = 64;
    while (seg > 8 && (long long)nlb * ((nal + seg - 1) / seg) < 152 * 32) seg /= 2;
    const int nseg = (nal + seg - 1) / seg;
    seg = (nal + nseg - 1) / nseg;
    if (D.d == 1) mb3::k3_march<T, 1><<<nlb * (unsigned)nseg, 32, 0, st>>>(D, seg, nlb);
    else mb3::k3_march<T, 2><<<nlb * (unsigned)nseg, 32, 0, st>>>(D, seg, nlb);
}
static void line_sweep(const Desc &D, bool near, cudaStream_t st) {
    if (D.f32) line_sweep_t<float>(D, near, st);
    else line_sweep_t<double>(D, near, st);
}
}

// one sweep's work on the streams, its report into slot `slot`, nothing
// waited for (nothing of the queue depends on a result on the host)
static mb_status queue_sweep(mb3_sim *s, int d, double dt, int slot) {
    cudaError_t e = cudaSuccess;
    const double delta = s->D.U[d] * dt;
    double TA[3] = {s->T[0], s->T[1], s->T[2]}, TM[3] = {TA[0], TA[1], TA[2]}, TB[3] = {TA[0], TA[1], TA[2]};
    TB[d] += delta;
    TM[d] += 0.5 * delta;
    int r0[3], rn[3];
    region(s, TA, TB, r0, rn);
    const size_t rc = (size_t)rn[0] * rn[1] * rn[2];
    const size_t rf = (size_t)(rn[0] + 1) * (rn[1] + 1) * (rn[2] + 1);
    if (e == cudaSuccess) e = ensure_r(s, rc, rf);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_sweep buffers");
    // pose A is the last pose computed (the previous sweep's B, or the pose
    // of the last state write or read): its fractions move to aP
    const bool reuse = s->prev_ok;
    if (reuse) {
        std::swap(s->D.aB, s->D.aP);
        std::swap(s->D.tB, s->D.tP);
        for (int a = 0; a < 3; ++a) { s->D.p0[a] = s->q0[a]; s->D.pn[a] = s->qn[a]; }
    }
    s->prev_ok = false;
    // three state buffers rotate: the step-start state stays in its own (Qn),
    // each sweep writes the new state into the free one (Cn)
    if (s->sidx == 0) s->dt_step = dt;
    Desc D = s->D;
    if (s->sidx == 0) D.Qn = D.Q;
    for (int a = 0; a < 3; ++a) { D.r0[a] = r0[a]; D.rn[a] = rn[a]; }
    D.d = d;
    D.lam = dt / D.h[d];
    D.hlam = 0.5 * D.lam;
    D.hlamf = 0.5f * (float)D.lam;
    if (e == cudaSuccess) e = cudaMemsetAsync(s->dev_report, 0, offsetof(mb3_sim::Report, err), s->st);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_sweep");
    const mb3::Body3 BA = posed(s, TA), BM = posed(s, TM), BB = posed(s, TB);
    if (rc > 0) {
        // the three geometry kernels are independent (each writes its own
        // arrays); the cut cells near a body's corners make each of them a
        // long tail on few SMs, so they run side by side on three streams,
        // and beside the cells that need no body data
        cudaEventRecord(s->fork, s->st);
        for (int q = 0; q < 3; ++q) cudaStreamWaitEvent(s->gs[q], s->fork, 0);
        mb3::k3_cells<<<nblk(32LL * (reuse ? 2 : 3) * (long long)rc), 256, 0, s->gs[0]>>>(
            D, BA, BM, BB, reuse ? mb3::CELLS_REUSE_A : mb3::CELLS_ALL);
        long long nfaces = 0;
        for (int a = 0; a < 4; ++a) {
            const int ax = a < 3 ? a : d;
            nfaces += (long long)(rn[0] + (ax == 0)) * (rn[1] + (ax == 1)) * (rn[2] + (ax == 2));
        }
        mb3::k3_faces<<<nblk(nfaces), 256, 0, s->gs[1]>>>(D, BM, BA, delta);
        if (delta != 0.0) {
            const long long nsw = (long long)(rn[0] + (d == 0)) * (rn[1] + (d == 1)) * (rn[2] + (d == 2));
            mb3::k3_swept<<<nblk(32LL * nsw), 256, 0, s->gs[2]>>>(D, BA, delta);
        }
        for (int q = 1; q < 3; ++q) {
            cudaEventRecord(s->join[q], s->gs[q]);
            cudaStreamWaitEvent(s->gs[0], s->join[q], 0);
        }
        mb3::k3_wall<<<nblk((long long)rc), 256, 0, s->gs[0]>>>(D);
        cudaEventRecord(s->join[0], s->gs[0]);
    }
    cudaEventRecord(s->ev[0], s->st);
    line_sweep(D, false, s->st);
    cudaEventRecord(s->ev[1], s->st);
    if (rc > 0) {
        cudaStreamWaitEvent(s->st, s->join[0], 0);
        cudaEventRecord(s->ev[2], s->st);
        line_sweep(D, true, s->st);
        cudaEventRecord(s->ev[3], s->st);
        mb3::k3_evprep<<<nblk((long long)rc), 256, 0, s->st>>>(D);
        mb3::k3_events<<<nblk((long long)rc), 256, 0, s->st>>>(D);
        mb3::k3_bad<<<nblk((long long)rc), 256, 0, s->st>>>(D);
    }
    mb3::k3_mix<<<1, mb3::MIXS_THREADS, 0, s->st>>>(D);
    if (rc > 0) mb3::k3_final<<<nblk((long long)rc), 256, 0, s->st>>>(D);
    // the new state's buffer becomes the state's; the next sweep writes into
    // the one left over
    s->D.Cn = s->sidx == 0 ? s->D.Qn : D.Q;
    s->D.Qn = D.Qn;
    s->D.Q = D.Cn;
    std::swap(s->D.Qf, s->D.Qfn);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(s->report + slot, s->dev_report, sizeof(mb3_sim::Report), cudaMemcpyDeviceToHost, s->st);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_sweep");
    s->prev_ok = true;
    for (int a = 0; a < 3; ++a) { s->q0[a] = r0[a]; s->qn[a] = rn[a]; }
    s->near_timed = rc > 0;
    s->T[d] = TB[d];
    if (++s->sidx == 3) {
        s->sidx = 0;
        s->t += dt;
        s->step++;
    }
    return MB_OK;
}
// waits for the queued sweeps whose reports go to slots 0 .. n-1; the status
// of the first that failed
static mb_status finish_sweeps(mb3_sim *s, int n) {
    const cudaError_t e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) {
        s->prev_ok = false;
        return cuda3(s, e, "mb3_sweep");
    }
    float far_ms = 0.0f, near_ms = 0.0f;
    cudaEventElapsedTime(&far_ms, s->ev[0], s->ev[1]);
    if (s->near_timed) cudaEventElapsedTime(&near_ms, s->ev[2], s->ev[3]);
    s->flux_ms = far_ms + near_ms;
    s->last_report = n - 1;
    mb_status first = MB_OK;
    for (int m = 0; m < n; ++m) {
        const mb_status r = err_status(s, s->report[m].err);
        if (first == MB_OK) first = r;
    }
    return first;
}

mb_status mb3_sweep(mb3_sim *s, int d, double dt) {
    if (!s || d < 0 || d > 2 || !(dt > 0.0)) return MB_E_INVAL;
    if (s->sidx > 0 && dt != s->dt_step) return fail3(s, MB_E_STATE, "the sweeps of a step must share dt");
    const mb_status r = queue_sweep(s, d, dt, 0);
    return r != MB_OK ? r : finish_sweeps(s, 1);
}

mb_status mb3_cfl_dt(mb3_sim *s, double *dt) {
    if (!s || !dt) return MB_E_INVAL;
    double *sm = s->smax_host;
    cudaError_t e = cudaMemsetAsync(s->D.smax, 0, 3 * sizeof(double), s->st);
    const unsigned nb = std::min(nblk(s->D.n), 152u * 8u);
    if (e == cudaSuccess && s->D.f32) mb3::k3_speeds32<<<nb, 256, 0, s->st>>>(s->D);
    else if (e == cudaSuccess)
        mb3::k3_speeds64<<<std::min(nblk(s->D.n, 256 * mb3::SPEED_CELLS), 152u * 8u), 256, 0, s->st>>>(s->D);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(sm, s->D.smax, 3 * sizeof(double), cudaMemcpyDeviceToHost, s->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_cfl_dt");
    double r = 1e300;
    for (int a = 0; a < 3; ++a) {
        double S = sm[a];
        if (s->nplane > 0) S = std::max(S, std::fabs(s->D.U[a]));
        if (S <= 0.0) S = 1e-300;
        r = std::min(r, s->D.h[a] / S);
    }
    *dt = s->cfl * r;
    return MB_OK;
}

mb_status mb3_step(mb3_sim *s, double dt, double *dt_used) {
    if (!s) return MB_E_INVAL;
    if (s->sidx != 0) return fail3(s, MB_E_STATE, "mb3_step in the middle of a step");
    if (!(dt > 0.0)) {
        const mb_status r = mb3_cfl_dt(s, &dt);
        if (r != MB_OK) return r;
    }
    if (dt_used) *dt_used = dt;
    if (!(dt > 0.0)) return MB_E_INVAL;
    // the three sweeps queued together: the host waits once per step
    const bool odd = s->step & 1;
    for (int m = 0; m < 3; ++m) {
        const mb_status r = queue_sweep(s, odd ? 2 - m : m, dt, m);
        if (r != MB_OK) {
            cudaStreamSynchronize(s->st);
            return r;
        }
    }
    return finish_sweeps(s, 3);
}

mb_status mb3_last_sweep(mb3_sim *s, double *wall, int *merged) {
    if (!s) return MB_E_INVAL;
    const mb3_sim::Report &r = s->report[s->last_report];
    if (wall) for (int q = 0; q < NC; ++q) wall[q] = r.wall[q];
    if (merged) *merged = r.mixed;
    return MB_OK;
}

mb_status mb3_set_precision(mb3_sim *s, int precision) {
    if (!s || (precision != MB_FP64 && precision != MB_FP32)) return MB_E_INVAL;
    if (s->sidx != 0) return fail3(s, MB_E_STATE, "mb3_set_precision in the middle of a step");
    cudaError_t e = cudaSuccess;
    if (precision == MB_FP32 && !s->D.Qf) e = dalloc(s, &s->D.Qf, NC * (size_t)s->D.n);
    if (e == cudaSuccess && precision == MB_FP32 && !s->D.Qfn) e = dalloc(s, &s->D.Qfn, NC * (size_t)s->D.n);
    if (e != cudaSuccess) return cuda3(s, e, "mb3_set_precision");
    s->D.f32 = precision == MB_FP32;
    if (s->D.f32) mb3::k3_to_f32<<<nblk(s->D.n), 256, 0, s->st>>>(s->D);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    return cuda3(s, e, "mb3_set_precision");
}

mb_status mb3_flux_time(mb3_sim *s, double *ms) {
    if (!s || !ms) return MB_E_INVAL;
    *ms = s->flux_ms;
    return MB_OK;
}

}  // extern "C"
