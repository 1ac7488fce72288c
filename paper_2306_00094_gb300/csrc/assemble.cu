// Assembly of the subdomain stiffness matrices A^k (FP64) on the GPU.
//
// A^k_ij = sum over ordered element pairs (E, E') inside Omega-hat_k u Gamma^D_k of
//   zeta(E,E')^-1 sum_q w_q |E| int_{E' cap B^h(x_q)} c(x_q, y) (psi_i(y)-psi_i(x_q)) (psi_j(y)-psi_j(x_q)) dy
// (eq. bilinear-multi1 with the quadrature of eq. bil1).  Rule (the same rule as
// the single-domain reference, implemented here from its definition):
//   outer points: 1-D 4-point Gauss-Legendre, 2-D 7-point degree-5 rule on E;
//   inner region: 1-D interval, 2-D l-infinity square clip, or the l2 "nocaps" polygon
//     (vertices of E' in the closed disc plus edge/circle crossings, Fig. approximate-ball e),
//     the "approxcaps" polygon (nocaps plus a chord/arc-midpoint triangle per left-out cap,
//     Fig. approximate-ball f), or, for the whole-element approximate balls (Fig. approximate-ball a-d), all of E'
//     when its barycenter / at least one vertex / at least two vertices lie in the disc;
//   constant kernels: exact polygon moments;
//   fractional / peridynamic kernels: if the bounding boxes of E and E' touch, polar
//     coordinates about x_q with the radial integral in closed form and 8-point
//     Gauss-Legendre in the angle on pieces (split at the edge normal, then each piece
//     ending half-way to +-pi/2); otherwise the 7-point rule on each fan triangle of
//     the polygon.
// On an inner element, psi_i(y) - psi_i(x) = a_i + g_i . (y - x) with g_i the gradient
// of the inner basis and a_i its linear extension at x minus the outer value; the
// inner integral is then a_i a_j S0 + (a_i g_j + a_j g_i) . S1 + g_i^T S2 g_j with
// kernel moments S0, S1, S2 of the region (rank-4 tensors for the vector kernel).
//
// 2-D: the host sorts the unordered pairs {E, E'} into three lists -- touching (bounding boxes
// touch), whole (apart, and E and E' within delta of each other everywhere, so that every inner
// region is the whole element) and cut (the rest) -- and each list is its own launch, so that the
// threads of a warp follow the same branch of the rule.  A CTA takes ASM_PAIRS pairs with one
// thread per (pair, orientation, outer point): each thread forms the kernel moments of its inner
// region, then one thread per row of a pair's local matrix adds the 7 or 14 points' contributions
// in order and scatters the row, weighted by 1/zeta, into the lower triangle of every A^k holding
// the pair (FP64 atomics) and into the Dirichlet coupling block; a second kernel mirrors the lower
// triangle so every A^k is exactly symmetric.  What bounds it is FP64 arithmetic (1/64 of the FP32
// rate): the moments call the power function once per radius (r^-2s; not at all for s = 1/2) and
// sincos once per angle (the direction follows by rotation with the edge normal), and a row of the
// local matrix takes 3 FMAs per entry and point from the point's combined moments.  On the
// fractional kernel with h = 1/64, delta = 6.4 h, 4 x 4 parts, s = 1/2: 72 ms (38.0 for 79 k touching
// pairs, 26.4 for 1.35 M cut, 7.5 for 0.63 M whole), against 600 ms for one thread per pair with the
// power function at every radial moment and the local matrix in shared memory; s = 0.4 or 0.75: 136 ms
// (58.9, 60.6, 16.8), against 663.
// 1-D: one thread per pair.
#include <algorithm>
#include <cmath>

#include "internal.hpp"

namespace nlf {
namespace {

struct AsmArgs {
    const double *xy;
    const int32_t *elems;
    const int8_t *node_dir;
    const uint64_t *mask;     // mask_words words per element: bit k % 64 of word k / 64 = subdomain k
    int mask_words;
    const int32_t *pairs;     // 2 * npairs
    int64_t npairs;
    const int32_t *nodemap;   // K x n_nodes
    int64_t n_nodes;
    const SubdomainDesc *sd;
    double *A;
    double *AD;
    int dim, type, nc;
    double delta, s, c;
    int ball;                 // 0 nocaps, 1 barycenter, 2 123vertices, 3 23vertices, 4 approxcaps (2-D l2)
};

__device__ const double kGLt8[8] = {-0.9602898564975363, -0.7966664774136267, -0.5255324099163290,
                                    -0.1834346424956498, 0.1834346424956498,  0.5255324099163290,
                                    0.7966664774136267,  0.9602898564975363};
__device__ const double kGLw8[8] = {0.1012285362903763, 0.2223810344533745, 0.3137066458778873, 0.3626837833783620,
                                    0.3626837833783620, 0.3137066458778873, 0.2223810344533745, 0.1012285362903763};

struct Rule7 {
    double b[7][3];
    double w[7];
};

__device__ __forceinline__ void rule7(Rule7 &r) {
    const double q15 = sqrt(15.0);
    const double p1 = (6.0 - q15) / 21.0, p2 = (6.0 + q15) / 21.0;
    const double w1 = (155.0 - q15) / 1200.0, w2 = (155.0 + q15) / 1200.0;
    const double c1 = 1.0 - 2.0 * p1, c2 = 1.0 - 2.0 * p2;
    double B[7][3] = {{1.0 / 3.0, 1.0 / 3.0, 1.0 / 3.0}, {p1, p1, c1}, {p1, c1, p1}, {c1, p1, p1},
                      {p2, p2, c2}, {p2, c2, p2}, {c2, p2, p2}};
    for (int q = 0; q < 7; ++q) {
        for (int i = 0; i < 3; ++i) r.b[q][i] = B[q][i];
        r.w[q] = q == 0 ? 9.0 / 40.0 : (q < 4 ? w1 : w2);
    }
}

// moments of the kernel over the inner region relative to x
struct Mom {
    double s0;
    double s1[2];
    double s2[3];          // xx, xy, yy
    // vector kernel: T0[ab] (xx,xy,yy), T1[abc] (xxx,xxy,xyy,yyy), T2[abcd] (xxxx,xxxy,xxyy,xyyy,yyyy)
    double t0[3], t1[4], t2[5];
};

__device__ __forceinline__ void mom_zero(Mom &m) {
    m.s0 = 0;
    m.s1[0] = m.s1[1] = 0;
    for (int i = 0; i < 3; ++i) m.s2[i] = 0, m.t0[i] = 0;
    for (int i = 0; i < 4; ++i) m.t1[i] = 0;
    for (int i = 0; i < 5; ++i) m.t2[i] = 0;
}

// add weight * {1, xi, xi xi^T} (scalar kernels)
__device__ __forceinline__ void mom_add_scalar(Mom &m, double w, double ex, double ey) {
    m.s0 += w;
    m.s1[0] += w * ex;
    m.s1[1] += w * ey;
    m.s2[0] += w * ex * ex;
    m.s2[1] += w * ex * ey;
    m.s2[2] += w * ey * ey;
}

// add sum over a direction: f0 th th^T + f1 th th^T th + f2 th th^T th th^T (vector kernel)
__device__ __forceinline__ void mom_add_vec(Mom &m, double f0, double f1, double f2, double cx, double cy) {
    double xx = cx * cx, xy = cx * cy, yy = cy * cy;
    m.t0[0] += f0 * xx; m.t0[1] += f0 * xy; m.t0[2] += f0 * yy;
    m.t1[0] += f1 * xx * cx; m.t1[1] += f1 * xx * cy; m.t1[2] += f1 * xy * cy; m.t1[3] += f1 * yy * cy;
    m.t2[0] += f2 * xx * xx; m.t2[1] += f2 * xx * xy; m.t2[2] += f2 * xx * yy; m.t2[3] += f2 * xy * yy;
    m.t2[4] += f2 * yy * yy;
}

__device__ __forceinline__ double tri_cross(const double *a, const double *b, const double *c) {
    return (b[0] - a[0]) * (c[1] - a[1]) - (b[1] - a[1]) * (c[0] - a[0]);
}

// ---------------------------------------------------------------- region construction
#define MAXV 12

__device__ int clip_axis(double (*P)[2], int n, int ax, double bound, double sgn) {
    double Q[MAXV][2];
    int m = 0;
    for (int k = 0; k < n; ++k) {
        const double *A = P[k], *B = P[(k + 1) % n];
        double fa = sgn * (A[ax] - bound), fb = sgn * (B[ax] - bound);
        if (fa <= 0.0) { Q[m][0] = A[0]; Q[m][1] = A[1]; ++m; }
        if ((fa < 0.0 && fb > 0.0) || (fa > 0.0 && fb < 0.0)) {
            double t = fa / (fa - fb);
            Q[m][0] = A[0] + t * (B[0] - A[0]);
            Q[m][1] = A[1] + t * (B[1] - A[1]);
            ++m;
        }
    }
    for (int k = 0; k < m; ++k) { P[k][0] = Q[k][0]; P[k][1] = Q[k][1]; }
    return m;
}

__device__ int region_square(const double (*T)[2], double x0, double x1, double d, double (*P)[2]) {
    for (int k = 0; k < 3; ++k) { P[k][0] = T[k][0]; P[k][1] = T[k][1]; }
    int n = clip_axis(P, 3, 0, x0 + d, 1.0);
    if (n) n = clip_axis(P, n, 0, x0 - d, -1.0);
    if (n) n = clip_axis(P, n, 1, x1 + d, 1.0);
    if (n) n = clip_axis(P, n, 1, x1 - d, -1.0);
    return n >= 3 ? n : 0;
}

// whole-element approximate ball: T itself when selected by the rule, else nothing
__device__ int region_whole(const double (*T)[2], double x0, double x1, double d, int ball, double (*P)[2]) {
    const double rr = d * d;
    int in = 0;
    for (int k = 0; k < 3; ++k) {
        const double dx = T[k][0] - x0, dy = T[k][1] - x1;
        if (dx * dx + dy * dy <= rr) ++in;
    }
    bool take;
    if (ball == 1) {
        const double bx = (T[0][0] + T[1][0] + T[2][0]) / 3.0 - x0, by = (T[0][1] + T[1][1] + T[2][1]) / 3.0 - x1;
        take = bx * bx + by * by <= rr;
    } else {
        take = in >= (ball == 2 ? 1 : 2);
    }
    if (!take) return 0;
    for (int k = 0; k < 3; ++k) {
        P[k][0] = T[k][0];
        P[k][1] = T[k][1];
    }
    return 3;
}

// l2 disc: the vertices of T in the closed disc and the edge/circle crossings strictly
// inside the edges, in boundary order ("nocaps").  With caps, every crossing where the
// boundary leaves the disc (the larger root on its edge) is followed by the point of the
// circle half-way along the arc to the next listed point, x + d (m - x) / |m - x| with m the
// chord midpoint ("approxcaps": each left-out cap becomes the triangle on its chord and arc
// midpoint; a minor arc, inside T, when 2 d exceeds the diameter of T).  At most 9 points:
// an edge adds its start vertex and one crossing, or two crossings, plus one arc point.
__device__ int region_disc(const double (*T)[2], double x0, double x1, double d, bool caps, double (*P)[2]) {
    int n = 0;
    const double rr = d * d;
    bool ex[MAXV];
    for (int k = 0; k < 3; ++k) {
        const double *A = T[k], *B = T[(k + 1) % 3];
        double px = A[0] - x0, py = A[1] - x1, ex_ = B[0] - A[0], ey = B[1] - A[1];
        double aa = px * px + py * py;
        if (aa <= rr) { P[n][0] = A[0]; P[n][1] = A[1]; ex[n] = false; ++n; }
        double qa = ex_ * ex_ + ey * ey, qb = px * ex_ + py * ey, qc = aa - rr;
        double disc = qb * qb - qa * qc;
        if (disc > 0.0) {
            double sq = sqrt(disc);
            double ta = (-qb - sq) / qa, tb = (-qb + sq) / qa;
            if (ta > 0.0 && ta < 1.0) { P[n][0] = A[0] + ta * ex_; P[n][1] = A[1] + ta * ey; ex[n] = false; ++n; }
            if (tb > 0.0 && tb < 1.0) { P[n][0] = A[0] + tb * ex_; P[n][1] = A[1] + tb * ey; ex[n] = true; ++n; }
        }
    }
    if (!caps) return n >= 3 ? n : 0;
    if (n < 2) return 0;
    // insert the arc points from the back, so that each lands after its exit crossing
    int m = n;
    for (int k = 0; k < n; ++k) m += ex[k] ? 1 : 0;
    const double qx = P[0][0], qy = P[0][1];      // the point after the last one
    int w = m;
    for (int k = n - 1; k >= 0; --k) {
        if (ex[k]) {
            const double nx = (k + 1 < n) ? P[k + 1][0] : qx, ny = (k + 1 < n) ? P[k + 1][1] : qy;
            double mx = 0.5 * (P[k][0] + nx) - x0, my = 0.5 * (P[k][1] + ny) - x1;
            double r = sqrt(mx * mx + my * my);
            if (r > 0.0) {
                --w;
                P[w][0] = x0 + d * mx / r;
                P[w][1] = x1 + d * my / r;
            } else {
                --m;            // a chord through x (not possible when 2 d > diam T): no arc point
            }
        }
        --w;
        P[w][0] = P[k][0];
        P[w][1] = P[k][1];
    }
    // w is 0 unless arc points were dropped; close the gap
    if (w > 0)
        for (int k = 0; k < m; ++k) { P[k][0] = P[k + w][0]; P[k][1] = P[k + w][1]; }
    return m >= 3 ? m : 0;
}

// exact moments of a polygon about x (constant kernel), by fan triangles:
// int_T 1 = |T|, int_T xi = |T| centroid, int_T xi xi^T = |T|/12 (sum v v^T + (sum v)(sum v)^T)
__device__ void moments_polygon(const double (*P)[2], int n, double x0, double x1, double c, Mom &m) {
    for (int k = 1; k + 1 < n; ++k) {
        double v[3][2] = {{P[0][0] - x0, P[0][1] - x1}, {P[k][0] - x0, P[k][1] - x1}, {P[k + 1][0] - x0, P[k + 1][1] - x1}};
        double at = 0.5 * ((v[1][0] - v[0][0]) * (v[2][1] - v[0][1]) - (v[1][1] - v[0][1]) * (v[2][0] - v[0][0]));
        double sx = v[0][0] + v[1][0] + v[2][0], sy = v[0][1] + v[1][1] + v[2][1];
        double qxx = v[0][0] * v[0][0] + v[1][0] * v[1][0] + v[2][0] * v[2][0] + sx * sx;
        double qxy = v[0][0] * v[0][1] + v[1][0] * v[1][1] + v[2][0] * v[2][1] + sx * sy;
        double qyy = v[0][1] * v[0][1] + v[1][1] * v[1][1] + v[2][1] * v[2][1] + sy * sy;
        double w = c * at;
        m.s0 += w;
        m.s1[0] += w * sx / 3.0;
        m.s1[1] += w * sy / 3.0;
        m.s2[0] += w * qxx / 12.0;
        m.s2[1] += w * qxy / 12.0;
        m.s2[2] += w * qyy / 12.0;
    }
}

// separated pair: 7-point rule on each fan triangle with the full kernel.  The kernel value at
// distance r from r^2: r^-(2+2s) = (r^2)^-(1+s), for s = 1/2 the cube of 1/r
__device__ void moments_fan7(const double (*P)[2], int n, double x0, double x1, const AsmArgs &a, const Rule7 &R,
                             Mom &m) {
    const double ax = P[0][0] - x0, ay = P[0][1] - x1;
    double bx = P[1][0] - x0, by = P[1][1] - x1;
    for (int k = 1; k + 1 < n; ++k) {
        const double cx = P[k + 1][0] - x0, cy = P[k + 1][1] - x1;
        const double wt = 0.5 * ((bx - ax) * (cy - ay) - (by - ay) * (cx - ax)) * a.c;
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            const double ex = R.b[q][0] * ax + R.b[q][1] * bx + R.b[q][2] * cx;
            const double ey = R.b[q][0] * ay + R.b[q][1] * by + R.b[q][2] * cy;
            const double r2 = ex * ex + ey * ey, w = wt * R.w[q];
            if (a.type == NLFETI_K_FRACTIONAL) {
                double f;
                if (a.s == 0.5) {
                    const double ri = rsqrt(r2);
                    f = w * (ri * ri * ri);
                } else {
                    f = w * pow(r2, -1.0 - a.s);
                }
                mom_add_scalar(m, f, ex, ey);
            } else {
                const double ri = rsqrt(r2), f = w * (ri * ri * ri);      // c xi xi^T / r^3
                const double fxx = f * ex * ex, fxy = f * ex * ey, fyy = f * ey * ey;
                m.t0[0] += fxx; m.t0[1] += fxy; m.t0[2] += fyy;
                m.t1[0] += fxx * ex; m.t1[1] += fxx * ey; m.t1[2] += fyy * ex; m.t1[3] += fyy * ey;
                m.t2[0] += fxx * ex * ex; m.t2[1] += fxx * ex * ey; m.t2[2] += fxx * ey * ey;
                m.t2[3] += fyy * ex * ey; m.t2[4] += fyy * ey * ey;
            }
        }
        bx = cx; by = cy;
    }
}

// touching pair: polar rule about x with the geometric angular split.  Along direction
// (cos, sin)(phi + ps), phi the angle of the edge normal (nx, ny), the radius is h / cos(ps) and
// the direction is the normal turned by ps
__device__ void moments_polar(const double (*P)[2], int n, double x0, double x1, const AsmArgs &a, Mom &m) {
    const double HALF_PI = 1.5707963267948966;
    const double e0 = -2.0 * a.s, e1 = 1.0 - 2.0 * a.s, e2 = 2.0 - 2.0 * a.s;     // radial exponents
    const bool half = a.s == 0.5, log1 = fabs(e1) < 1e-14;
    const double i0 = 1.0 / e0, i1 = log1 ? 0.0 : 1.0 / e1, i2 = 1.0 / e2;
    for (int k = 0; k < n; ++k) {
        const int k1 = k + 1 < n ? k + 1 : 0;
        double ux = P[k][0] - x0, uy = P[k][1] - x1;
        double vx = P[k1][0] - x0, vy = P[k1][1] - x1;
        double ex = vx - ux, ey = vy - uy;
        double len = sqrt(ex * ex + ey * ey);
        if (len == 0.0) continue;
        double nx = ey / len, ny = -ex / len;
        double h = nx * ux + ny * uy;
        if (h < 0.0) { nx = -nx; ny = -ny; h = -h; }
        if (h <= 0.0) continue;
        double au = atan2(nx * uy - ny * ux, nx * ux + ny * uy);
        double av = atan2(nx * vy - ny * vx, nx * vx + ny * vy);
        const double sg = av >= au ? a.c : -a.c;
        double lo = fmin(au, av), hi = fmax(au, av);
        // pieces: [lo,0],[0,hi] if straddling, each subdivided toward +-pi/2
        double seg[2][2];
        int nseg;
        if (lo < 0.0 && hi > 0.0) { seg[0][0] = lo; seg[0][1] = 0.0; seg[1][0] = 0.0; seg[1][1] = hi; nseg = 2; }
        else { seg[0][0] = lo; seg[0][1] = hi; nseg = 1; }
        int count = 0;
        for (int sgi = 0; sgi < nseg; ++sgi) {
            bool neg = seg[sgi][1] <= 0.0;
            double cur = neg ? -seg[sgi][1] : seg[sgi][0];
            double end = neg ? -seg[sgi][0] : seg[sgi][1];
            while (cur < end && count < 64) {
                double nxt = 0.5 * (cur + HALF_PI);
                if (nxt >= end || count == 63) nxt = end;
                double pa = neg ? -nxt : cur, pb = neg ? -cur : nxt;
                ++count;
                const double hw = 0.5 * (pb - pa);
                for (int t = 0; t < 8; ++t) {
                    const double ps = pa + hw * (1.0 + kGLt8[t]);
                    double sp, cp;
                    sincos(ps, &sp, &cp);
                    const double cth = nx * cp - ny * sp, sth = ny * cp + nx * sp;
                    const double rho = h / cp, W = hw * kGLw8[t] * sg;
                    if (a.type == NLFETI_K_FRACTIONAL) {
                        const double rp = half ? cp / h : pow(rho, e0);           // rho^-2s
                        const double r1 = W * (log1 ? log(rho) : rp * rho * i1), r2 = W * (rp * rho * rho * i2);
                        m.s0 += W * (rp * i0);
                        m.s1[0] += r1 * cth;
                        m.s1[1] += r1 * sth;
                        m.s2[0] += r2 * cth * cth;
                        m.s2[1] += r2 * cth * sth;
                        m.s2[2] += r2 * sth * sth;
                    } else {
                        mom_add_vec(m, W * rho, W * 0.5 * rho * rho, W * rho * rho * rho / 3.0, cth, sth);
                    }
                }
                cur = nxt;
            }
        }
    }
}

// scatter row p (component rp of the subdomain's row map) of a pair's local matrix into every
// subdomain holding the pair: v[q], q < ld, weighted by 1/zeta
template <int NC>
__device__ __forceinline__ void scatter_row(const AsmArgs &a, int E0, int E1, const int *nodes, int ld, int p,
                                            const double *v) {
    int zeta = 0;
    for (int w = 0; w < a.mask_words; ++w)
        zeta += __popcll(a.mask[(int64_t)E0 * a.mask_words + w] & a.mask[(int64_t)E1 * a.mask_words + w]);
    const double wz = 1.0 / (double)zeta;
    for (int w = 0; w < a.mask_words; ++w) {
        uint64_t both = a.mask[(int64_t)E0 * a.mask_words + w] & a.mask[(int64_t)E1 * a.mask_words + w];
        while (both) {
            const int k = 64 * w + __ffsll((long long)both) - 1;
            both &= both - 1;
            const int32_t *map = a.nodemap + (int64_t)k * a.n_nodes;
            const int mp = map[nodes[p / NC]];
            if (mp < 0) continue;
            const SubdomainDesc &d = a.sd[k];
            const int rp = mp * NC + p % NC;
            double *Arow = a.A + d.offA + (int64_t)rp * d.nk, *ADrow = a.AD + d.offAD + (int64_t)rp * d.nD;
#pragma unroll
            for (int q = 0; q < 6 * NC; ++q) {
                if (q >= ld) continue;
                const int mq = map[nodes[q / NC]];
                if (mq >= 0) {
                    const int cq = mq * NC + q % NC;
                    if (rp >= cq) atomicAdd(Arow + cq, wz * v[q]);
                } else if (mq <= -2) {
                    atomicAdd(ADrow + (-2 - mq) * NC + q % NC, wz * v[q]);
                }
            }
        }
    }
}

// 1-D: one thread per unordered pair, both orientations
__global__ void __launch_bounds__(64) k_assemble_1d(AsmArgs a) {
    const int64_t pid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pid >= a.npairs) return;
    const int E0 = a.pairs[2 * pid], E1 = a.pairs[2 * pid + 1];
    int nodes[6];
    int nl = 0;
    for (int i = 0; i < 2; ++i) nodes[nl++] = a.elems[2 * (int64_t)E0 + i];
    for (int i = 0; i < 2; ++i) {
        const int nd = a.elems[2 * (int64_t)E1 + i];
        if (nodes[0] != nd && nodes[1] != nd) nodes[nl++] = nd;
    }
    double acc[4][6];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 6; ++j) acc[i][j] = 0.0;
    const double q1 = sqrt(3.0 / 7.0 - 2.0 / 7.0 * sqrt(6.0 / 5.0)), q2 = sqrt(3.0 / 7.0 + 2.0 / 7.0 * sqrt(6.0 / 5.0));
    const double w1 = (18.0 + sqrt(30.0)) / 36.0, w2 = (18.0 - sqrt(30.0)) / 36.0;
    const double tq[4] = {-q2, -q1, q1, q2}, wq[4] = {w2, w1, w1, w2};
    const int ndir = (E0 == E1) ? 1 : 2;
    for (int dir = 0; dir < ndir; ++dir) {
        const int Eo = dir == 0 ? E0 : E1, Ei = dir == 0 ? E1 : E0;
        const int no0 = a.elems[2 * (int64_t)Eo], no1 = a.elems[2 * (int64_t)Eo + 1];
        const int ni0 = a.elems[2 * (int64_t)Ei], ni1 = a.elems[2 * (int64_t)Ei + 1];
        const double o0 = a.xy[no0], o1 = a.xy[no1], i0 = a.xy[ni0], i1 = a.xy[ni1];
        const double hin = i1 - i0;
        double g[4];
        for (int i = 0; i < nl; ++i) g[i] = nodes[i] == ni0 ? -1.0 / hin : (nodes[i] == ni1 ? 1.0 / hin : 0.0);
        for (int q = 0; q < 4; ++q) {
            const double lam = 0.5 * (1.0 + tq[q]);
            const double x = o0 + (o1 - o0) * lam;
            const double lo = fmax(fmin(i0, i1), x - a.delta), hi = fmin(fmax(i0, i1), x + a.delta);
            if (!(hi > lo)) continue;
            double av[4];
            for (int i = 0; i < nl; ++i) {
                const double outv = nodes[i] == no0 ? 1.0 - lam : (nodes[i] == no1 ? lam : 0.0);
                const double inv = nodes[i] == ni0 ? (i1 - x) / hin : (nodes[i] == ni1 ? (x - i0) / hin : 0.0);
                av[i] = (Eo == Ei) ? 0.0 : inv - outv;
            }
            const double dl = lo - x, dh = hi - x;
            const double s0 = a.c * (dh - dl), s1 = a.c * 0.5 * (dh * dh - dl * dl),
                         s2 = a.c * (dh * dh * dh - dl * dl * dl) / 3.0, wt = 0.5 * wq[q] * fabs(o1 - o0);
            for (int i = 0; i < nl; ++i)
                for (int j = 0; j < nl; ++j)
                    acc[i][j] += wt * (av[i] * av[j] * s0 + (av[i] * g[j] + av[j] * g[i]) * s1 + g[i] * g[j] * s2);
        }
    }
    for (int i = 0; i < nl; ++i) scatter_row<1>(a, E0, E1, nodes, nl, i, acc[i]);
}

// the bounding boxes of the outer and the inner element touch (relative to the outer one's size)
__device__ __forceinline__ bool boxes_touch(const double (*To)[2], const double (*Ti)[2]) {
    double gap = 0.0, ext = 0.0;
    for (int c = 0; c < 2; ++c) {
        const double lo0 = fmin(fmin(To[0][c], To[1][c]), To[2][c]), hi0 = fmax(fmax(To[0][c], To[1][c]), To[2][c]);
        const double lo1 = fmin(fmin(Ti[0][c], Ti[1][c]), Ti[2][c]), hi1 = fmax(fmax(Ti[0][c], Ti[1][c]), Ti[2][c]);
        gap = fmax(gap, fmax(lo1 - hi0, lo0 - hi1));
        ext = fmax(ext, hi0 - lo0);
    }
    return gap <= 1e-9 * ext;
}

// 2-D.  CLS: the list the pairs come from (touching, cut, whole).  Shared memory holds, per pair
// (fastest index, so that the lanes of a warp read consecutive words): the geometry of its two
// orientations and, per (orientation, outer point), the weighted moments and the values a_i.
enum { ASM_TOUCH = 0, ASM_CUT = 1, ASM_WHOLE = 2 };
constexpr int ASM_PAIRS = 16;                     // pairs of a CTA
constexpr int ASM_THREADS = ASM_PAIRS * 14;       // (pair, orientation, outer point)
template <int NC> constexpr int asm_moments() { return NC == 1 ? 6 : 12; }
template <int NC> constexpr size_t asm_smem_bytes() {
    return sizeof(double) * ASM_PAIRS * (2 * 18 + 14 * (6 + asm_moments<NC>()));
}

template <int NC, int CLS>
__global__ void __launch_bounds__(ASM_THREADS) k_assemble(AsmArgs a) {
    extern __shared__ double smem[];
    constexpr int NM = asm_moments<NC>(), PB = ASM_PAIRS;
    double *geo = smem;                           // [orientation][i][gx, gy, l0][pair]
    double *avs = geo + 2 * 18 * PB;              // [orientation, point][i][pair]
    double *mom = avs + 14 * 6 * PB;              // [orientation, point][moment][pair]
    __shared__ int snodes[PB][6], snl[PB];
    __shared__ int8_t sio[2][PB][6];              // position of node i in the outer element, or -1
    const int64_t pid0 = (int64_t)blockIdx.x * PB;
    const int npb = (int)min((int64_t)PB, a.npairs - pid0);
    // the pair's nodes and, per orientation, the gradient and the value at the origin of the inner
    // linear functions: lambda_v(y) = cross(T[v+1]-y, T[v+2]-y) / Di
    if (threadIdx.x < 2 * PB && threadIdx.x % PB < npb) {
        const int pl = threadIdx.x % PB, dir = threadIdx.x / PB;
        const int E0 = a.pairs[2 * (pid0 + pl)], E1 = a.pairs[2 * (pid0 + pl) + 1];
        const int Eo = dir == 0 ? E0 : E1, Ei = dir == 0 ? E1 : E0;
        int nodes[6], nl = 0;
        for (int i = 0; i < 3; ++i) nodes[nl++] = a.elems[3 * (int64_t)E0 + i];
        for (int i = 0; i < 3; ++i) {
            const int nd = a.elems[3 * (int64_t)E1 + i];
            if (nodes[0] != nd && nodes[1] != nd && nodes[2] != nd) nodes[nl++] = nd;
        }
        int no[3], ni[3];
        double T[3][2];
        for (int v = 0; v < 3; ++v) {
            no[v] = a.elems[3 * (int64_t)Eo + v];
            ni[v] = a.elems[3 * (int64_t)Ei + v];
            T[v][0] = a.xy[2 * (int64_t)ni[v]];
            T[v][1] = a.xy[2 * (int64_t)ni[v] + 1];
        }
        const double Di = tri_cross(T[0], T[1], T[2]);
        for (int i = 0; i < 6; ++i) {
            int io = -1, ii = -1;
            for (int v = 0; v < 3; ++v) {
                if (i < nl && no[v] == nodes[i]) io = v;
                if (i < nl && ni[v] == nodes[i]) ii = v;
            }
            double gx = 0.0, gy = 0.0, l0 = 0.0;
            if (ii >= 0) {
                const double *P1 = T[(ii + 1) % 3], *P2 = T[(ii + 2) % 3];
                gx = (P1[1] - P2[1]) / Di;
                gy = (P2[0] - P1[0]) / Di;
                l0 = (P1[0] * P2[1] - P1[1] * P2[0]) / Di;
            }
            geo[((dir * 6 + i) * 3 + 0) * PB + pl] = gx;
            geo[((dir * 6 + i) * 3 + 1) * PB + pl] = gy;
            geo[((dir * 6 + i) * 3 + 2) * PB + pl] = l0;
            sio[dir][pl][i] = (int8_t)io;
            if (dir == 0) snodes[pl][i] = i < nl ? nodes[i] : -1;
        }
        if (dir == 0) snl[pl] = nl;
    }
    __syncthreads();
    // one thread per (pair, orientation, outer point): the moments of the inner region, weighted by
    // the outer rule, and a_i (0 for the pair of an element with itself)
    {
        const int pl = threadIdx.x % PB, dq = threadIdx.x / PB, dir = dq / 7, q = dq % 7;
        Mom m;
        mom_zero(m);
        double av[6] = {0, 0, 0, 0, 0, 0};
        double wt = 0.0;
        if (pl < npb) {
            const int E0 = a.pairs[2 * (pid0 + pl)], E1 = a.pairs[2 * (pid0 + pl) + 1];
            if (dir == 0 || E0 != E1) {
                const int Eo = dir == 0 ? E0 : E1, Ei = dir == 0 ? E1 : E0;
                Rule7 R;
                rule7(R);
                double To[3][2], Ti[3][2];
                for (int v = 0; v < 3; ++v) {
                    const int no = a.elems[3 * (int64_t)Eo + v], ni = a.elems[3 * (int64_t)Ei + v];
                    To[v][0] = a.xy[2 * (int64_t)no]; To[v][1] = a.xy[2 * (int64_t)no + 1];
                    Ti[v][0] = a.xy[2 * (int64_t)ni]; Ti[v][1] = a.xy[2 * (int64_t)ni + 1];
                }
                const double b0 = R.b[q][0], b1 = R.b[q][1], b2 = R.b[q][2];
                const double x0 = b0 * To[0][0] + b1 * To[1][0] + b2 * To[2][0];
                const double x1 = b0 * To[0][1] + b1 * To[1][1] + b2 * To[2][1];
                double P[MAXV][2];
                int np = 3;
                if (CLS == ASM_WHOLE) {
                    for (int v = 0; v < 3; ++v) { P[v][0] = Ti[v][0]; P[v][1] = Ti[v][1]; }
                } else {
                    np = (a.type == NLFETI_K_CONST_LINF) ? region_square(Ti, x0, x1, a.delta, P)
                         : (a.ball != 0 && a.ball != 4)   ? region_whole(Ti, x0, x1, a.delta, a.ball, P)
                                                          : region_disc(Ti, x0, x1, a.delta, a.ball == 4, P);
                }
                if (np > 0) {
                    wt = R.w[q] * 0.5 * fabs(tri_cross(To[0], To[1], To[2]));
                    if (NC == 1 && (a.type == NLFETI_K_CONST_LINF || a.type == NLFETI_K_CONST_L2))
                        moments_polygon(P, np, x0, x1, a.c, m);
                    else if (CLS == ASM_TOUCH && boxes_touch(To, Ti)) moments_polar(P, np, x0, x1, a, m);
                    else moments_fan7(P, np, x0, x1, a, R, m);
                    if (Eo != Ei)
                        for (int i = 0; i < 6; ++i) {
                            const int io = sio[dir][pl][i];
                            const double *gp = geo + (dir * 6 + i) * 3 * PB + pl;
                            const double outv = io == 0 ? b0 : (io == 1 ? b1 : (io == 2 ? b2 : 0.0));
                            av[i] = gp[2 * PB] + gp[0] * x0 + gp[PB] * x1 - outv;
                        }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) avs[(dq * 6 + i) * PB + pl] = av[i];
        double *mp = mom + dq * NM * PB + pl;
        if (NC == 1) {
            mp[0] = wt * m.s0;
            mp[PB] = wt * m.s1[0];
            mp[2 * PB] = wt * m.s1[1];
            for (int e = 0; e < 3; ++e) mp[(3 + e) * PB] = wt * m.s2[e];
        } else {
            for (int e = 0; e < 3; ++e) mp[e * PB] = wt * m.t0[e];
            for (int e = 0; e < 4; ++e) mp[(3 + e) * PB] = wt * m.t1[e];
            for (int e = 0; e < 5; ++e) mp[(7 + e) * PB] = wt * m.t2[e];
        }
    }
    __syncthreads();
    // one thread per (pair, row): row p of the local matrix, the points in order.  With
    //   a_i a_j S0 + (a_i g_j + a_j g_i) . S1 + g_i^T S2 g_j = a_j (a_i S0 + g_i . S1) + g_j . (a_i S1 + S2 g_i)
    // (vector kernel: component (al, be) takes the moments contracted with the unit vectors al, be)
    for (int t = threadIdx.x; t < PB * 6 * NC; t += ASM_THREADS) {
        const int pl = t % PB, p = t / PB, i = p / NC, al = p % NC;
        if (pl >= npb || i >= snl[pl]) continue;
        const int nl = snl[pl];
        double v[6 * NC];
#pragma unroll
        for (int e = 0; e < 6 * NC; ++e) v[e] = 0.0;
        for (int dir = 0; dir < 2; ++dir) {
            const double *gd = geo + dir * 18 * PB + pl;
            const double gix = gd[(3 * i) * PB], giy = gd[(3 * i + 1) * PB];
            for (int q = 0; q < 7; ++q) {
                const int dq = dir * 7 + q;
                const double *mp = mom + dq * NM * PB + pl, *ap = avs + dq * 6 * PB + pl;
                const double ai = ap[i * PB];
#pragma unroll
                for (int be = 0; be < NC; ++be) {
                    // moments of component (al, be): S0, S1 (x, y), S2 (xx, xy, yy)
                    double s0, s1x, s1y, sxx, sxy, syy;
                    if (NC == 1) {
                        s0 = mp[0]; s1x = mp[PB]; s1y = mp[2 * PB];
                        sxx = mp[3 * PB]; sxy = mp[4 * PB]; syy = mp[5 * PB];
                    } else {
                        const int o = al + be;
                        s0 = mp[o * PB]; s1x = mp[(3 + o) * PB]; s1y = mp[(4 + o) * PB];
                        sxx = mp[(7 + o) * PB]; sxy = mp[(8 + o) * PB]; syy = mp[(9 + o) * PB];
                    }
                    const double f0 = ai * s0 + gix * s1x + giy * s1y;
                    const double fx = ai * s1x + gix * sxx + giy * sxy, fy = ai * s1y + gix * sxy + giy * syy;
#pragma unroll
                    for (int j = 0; j < 6; ++j)
                        v[NC * j + be] += ap[j * PB] * f0 + gd[(3 * j) * PB] * fx + gd[(3 * j + 1) * PB] * fy;
                }
            }
        }
        scatter_row<NC>(a, a.pairs[2 * (pid0 + pl)], a.pairs[2 * (pid0 + pl) + 1], snodes[pl], nl * NC, p, v);
    }
}

__global__ void k_mirror(double *A, const SubdomainDesc *sd) {
    const SubdomainDesc d = sd[blockIdx.y];
    double *M = A + d.offA;
    const int64_t n = d.nk;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * n; t += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = t / n, j = t % n;
        if (j > i) M[t] = M[j * n + i];
    }
}

}  // namespace

void assemble_all(nlfeti_problem *p) {
    nlfeti_ctx *c = p->ctx;
    const MeshHost &m = p->mesh;
    // unordered pair list: bounding boxes within delta, sharing a subdomain, not both in the collar
    const int nv = m.dim + 1;
    std::vector<double> lo(m.n_elems * 2, 0.0), hi(m.n_elems * 2, 0.0);
    double ext = 0.0, glo[2] = {INFINITY, INFINITY}, ghi[2] = {-INFINITY, -INFINITY};
    for (int64_t e = 0; e < m.n_elems; ++e) {
        for (int a = 0; a < m.dim; ++a) { lo[2 * e + a] = INFINITY; hi[2 * e + a] = -INFINITY; }
        for (int i = 0; i < nv; ++i) {
            int32_t n = m.elems[e * nv + i];
            for (int a = 0; a < m.dim; ++a) {
                double x = m.xy[(int64_t)n * m.dim + a];
                lo[2 * e + a] = std::min(lo[2 * e + a], x);
                hi[2 * e + a] = std::max(hi[2 * e + a], x);
            }
        }
        for (int a = 0; a < m.dim; ++a) {
            ext = std::max(ext, hi[2 * e + a] - lo[2 * e + a]);
            glo[a] = std::min(glo[a], lo[2 * e + a]);
            ghi[a] = std::max(ghi[a], hi[2 * e + a]);
        }
    }
    const double H = ext > 0 ? ext : 1.0;
    int64_t nb[2] = {1, 1};
    for (int a = 0; a < m.dim; ++a) nb[a] = (int64_t)std::floor((ghi[a] - glo[a]) / H) + 1;
    std::vector<int64_t> start(nb[0] * nb[1] + 1, 0), items(m.n_elems), cell(m.n_elems);
    for (int64_t e = 0; e < m.n_elems; ++e) {
        int64_t cc[2] = {0, 0};
        for (int a = 0; a < m.dim; ++a)
            cc[a] = std::clamp<int64_t>((int64_t)std::floor((lo[2 * e + a] - glo[a]) / H), 0, nb[a] - 1);
        cell[e] = cc[1] * nb[0] + cc[0];
        start[cell[e] + 1]++;
    }
    for (size_t i = 0; i + 1 < start.size(); ++i) start[i + 1] += start[i];
    {
        std::vector<int64_t> fill(start.begin(), start.end() - 1);
        for (int64_t e = 0; e < m.n_elems; ++e) items[fill[cell[e]]++] = e;
    }
    const double r = p->kern.delta;
    // 2-D pair lists: touching, cut, whole (see the file comment; the bounding boxes decide, so a
    // pair of the cut list may still have whole regions); 1-D: one list
    std::vector<int32_t> pairs[3];
    for (auto &v : pairs) v.reserve(1 << 18);
    const bool square = p->kern.type == NLFETI_K_CONST_LINF;
    for (int64_t e = 0; e < m.n_elems; ++e) {
        if (!p->dec.any_sub(e)) continue;
        int64_t clo[2] = {0, 0}, chi[2] = {0, 0};
        for (int a = 0; a < m.dim; ++a) {
            clo[a] = std::max<int64_t>(0, (int64_t)std::floor((lo[2 * e + a] - r - H - glo[a]) / H) - 1);
            chi[a] = std::min<int64_t>(nb[a] - 1, (int64_t)std::floor((hi[2 * e + a] + r - glo[a]) / H) + 1);
        }
        for (int64_t cy = clo[1]; cy <= chi[1]; ++cy)
            for (int64_t cx = clo[0]; cx <= chi[0]; ++cx) {
                int64_t cidx = cy * nb[0] + cx;
                for (int64_t t = start[cidx]; t < start[cidx + 1]; ++t) {
                    int64_t f = items[t];
                    if (f < e) continue;
                    if (!p->dec.share_sub(e, f)) continue;
                    if (m.elem_dir[e] && m.elem_dir[f]) continue;
                    double gap = 0.0;
                    for (int a = 0; a < m.dim; ++a)
                        gap = std::max(gap, std::max(lo[2 * f + a] - hi[2 * e + a], lo[2 * e + a] - hi[2 * f + a]));
                    if (gap > r) continue;
                    int cls = ASM_TOUCH;
                    if (m.dim == 2) {
                        // the touching test is relative to the outer element's size (the kernel repeats it
                        // per orientation)
                        const double he = std::max(hi[2 * e] - lo[2 * e], hi[2 * e + 1] - lo[2 * e + 1]),
                                     hf = std::max(hi[2 * f] - lo[2 * f], hi[2 * f + 1] - lo[2 * f + 1]);
                        if (!(gap <= 1e-9 * std::max(he, hf))) {
                            const double wx = std::max(hi[2 * f] - lo[2 * e], hi[2 * e] - lo[2 * f]),
                                         wy = std::max(hi[2 * f + 1] - lo[2 * e + 1], hi[2 * e + 1] - lo[2 * f + 1]);
                            const bool whole = square ? std::max(wx, wy) <= r * (1.0 - 1e-12)
                                                      : wx * wx + wy * wy <= r * r * (1.0 - 1e-12);
                            cls = whole ? ASM_WHOLE : ASM_CUT;
                        }
                    }
                    pairs[cls].push_back((int32_t)e);
                    pairs[cls].push_back((int32_t)f);
                }
            }
    }
    DevMem d_pairs[3];
    for (int l = 0; l < 3; ++l)
        if (!pairs[l].empty()) upload(c, d_pairs[l], pairs[l]);
    NLF_CUDA(cudaMemsetAsync(p->d_A.p, 0, p->d_A.bytes, c->stream));
    NLF_CUDA(cudaMemsetAsync(p->d_AD.p, 0, p->d_AD.bytes, c->stream));
    AsmArgs a;
    a.xy = p->d_xy.as<double>();
    a.elems = p->d_elems.as<int32_t>();
    a.node_dir = p->d_node_dir.as<int8_t>();
    a.mask = p->d_elem_mask.as<uint64_t>();
    a.mask_words = p->dec.mask_words;
    a.nodemap = p->d_nodemap.as<int32_t>();
    a.n_nodes = m.n_nodes;
    a.sd = p->d_sd.as<SubdomainDesc>();
    a.A = p->d_A.as<double>();
    a.AD = p->d_AD.as<double>();
    a.dim = m.dim;
    a.type = p->kern.type;
    a.nc = p->nc;
    a.delta = p->kern.delta;
    a.ball = p->kern.ball;
    a.s = p->kern.s;
    a.c = p->kern.scale;
    auto launch = [&](auto kern, int l, int per_cta, int threads, size_t smem) {
        const int64_t npairs = (int64_t)pairs[l].size() / 2;
        if (smem > 48 * 1024)
            NLF_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const int64_t chunk = 1 << 24;     // keep the grid within limits
        for (int64_t off = 0; off < npairs; off += chunk) {
            AsmArgs b = a;
            b.pairs = d_pairs[l].as<int32_t>() + 2 * off;
            b.npairs = std::min<int64_t>(chunk, npairs - off);
            kern<<<(unsigned)((b.npairs + per_cta - 1) / per_cta), threads, smem, c->stream>>>(b);
            NLF_CUDA(cudaGetLastError());
        }
    };
    if (m.dim == 1) {
        launch(k_assemble_1d, ASM_TOUCH, 64, 64, 0);
    } else if (p->nc == 1) {
        launch(k_assemble<1, ASM_TOUCH>, ASM_TOUCH, ASM_PAIRS, ASM_THREADS, asm_smem_bytes<1>());
        launch(k_assemble<1, ASM_CUT>, ASM_CUT, ASM_PAIRS, ASM_THREADS, asm_smem_bytes<1>());
        launch(k_assemble<1, ASM_WHOLE>, ASM_WHOLE, ASM_PAIRS, ASM_THREADS, asm_smem_bytes<1>());
    } else {
        launch(k_assemble<2, ASM_TOUCH>, ASM_TOUCH, ASM_PAIRS, ASM_THREADS, asm_smem_bytes<2>());
        launch(k_assemble<2, ASM_CUT>, ASM_CUT, ASM_PAIRS, ASM_THREADS, asm_smem_bytes<2>());
        launch(k_assemble<2, ASM_WHOLE>, ASM_WHOLE, ASM_PAIRS, ASM_THREADS, asm_smem_bytes<2>());
    }
    dim3 grid(64, p->K);
    k_mirror<<<grid, 256, 0, c->stream>>>(p->d_A.as<double>(), p->d_sd.as<SubdomainDesc>());
    NLF_CUDA(cudaGetLastError());
    NLF_CUDA(cudaStreamSynchronize(c->stream));
}

}  // namespace nlf
