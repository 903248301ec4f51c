// lks_quad.cuh -- the FP64 step of a band (lks_resident.cuh) with four warps to a group of 32 nodes.
//
// An FP64 warp instruction holds its SM sub-partition's FP64 unit for 64 clocks, active lanes or not, so a warp
// that steps 32 nodes on its own needs 64 clocks for each of the collision's 104-114 instructions: 3.7 us, and a
// small lattice has no other warps to fill the SM with.  Four warps, one per sub-partition, split the work:
// first the moments (rho and 3/rho; j_x; j_y; B), exchanged through shared memory, then the populations (f1 f3;
// f0 f2 f4; f5..8; g), with the few common terms computed by each.  Per group the longest chain is 46
// instructions.  A 4 x 65 channel takes 2.3 us a step, with one warp to 32 nodes 4.3, in single-step kernels 5.0.
// Every operation is collide_pairs' own, so are the bits.  Maxwell coupling.
#pragma once
#include "lks_resident.cuh"

namespace lks {

constexpr int kQuadWords = 7 * 32;  // doubles of shared memory per group: drho, 3/rho, jx, jy, bx, dby, by

template <int CLOSURE, bool FORCE>
__device__ __forceinline__ void quad_step(const Band<double>& band, int b, const StepParams<double>& p, double* sh) {
    const int role = (threadIdx.x >> 5) & 3, quad = threadIdx.x >> 7, lane = threadIdx.x & 31;
    const int nx = band.nx, plane = band.plane, nodes = band.rows * nx;
    const bool active = quad * 32 + lane < nodes;
    const int node = active ? quad * 32 + lane : 0;
    const int jl = node / nx, i = node - jl * nx, j = band.first + jl;
    const bool bottom = j == 0, top = j == p.ny - 1;
    const int rc = (jl + 1) * nx, rs = rc - nx, rn = rc + nx;
    const int im = i == 0 ? nx - 1 : i - 1, ip = i == nx - 1 ? 0 : i + 1;
    const double* in = band.buf(b);
    double* out = band.buf(b ^ 1);
    double* q = sh + quad * kQuadWords + lane;
    double f[9], gx[5], gy[5];

    // the pulls and link closures of step_node_with
    auto load_f = [&]() {
        const double* u = in;
        f[0] = u[0 * plane + rc + i];
        f[1] = u[1 * plane + rc + im];
        f[3] = u[3 * plane + rc + ip];
        if (!bottom) {
            f[2] = u[2 * plane + rs + i];
            f[5] = u[5 * plane + rs + im];
            f[6] = u[6 * plane + rs + ip];
        } else if (CLOSURE == 0) {
            f[2] = u[4 * plane + rc + i];
            f[5] = u[7 * plane + rc + i] + p.bot.du;
            f[6] = u[8 * plane + rc + i] - p.bot.du;
        }
        if (!top) {
            f[4] = u[4 * plane + rn + i];
            f[7] = u[7 * plane + rn + ip];
            f[8] = u[8 * plane + rn + im];
        } else if (CLOSURE == 0) {
            f[4] = u[2 * plane + rc + i];
            f[7] = u[5 * plane + rc + i] - p.top.du;
            f[8] = u[6 * plane + rc + i] + p.top.du;
        }
    };
    auto load_g = [&]() {
        const double *u = in + 9 * plane, *v = in + 14 * plane;
        gx[0] = u[0 * plane + rc + i];
        gx[1] = u[1 * plane + rc + im];
        gx[3] = u[3 * plane + rc + ip];
        gy[0] = v[0 * plane + rc + i];
        gy[1] = v[1 * plane + rc + im];
        gy[3] = v[3 * plane + rc + ip];
        if (!bottom) {
            gx[2] = u[2 * plane + rs + i];
            gy[2] = v[2 * plane + rs + i];
        } else if (CLOSURE == 0) {
            gx[2] = ffma(p.bot.r, u[4 * plane + rc + i], p.bot.kx);
            gy[2] = -v[4 * plane + rc + i];
        }
        if (!top) {
            gx[4] = u[4 * plane + rn + i];
            gy[4] = v[4 * plane + rn + i];
        } else if (CLOSURE == 0) {
            gx[4] = ffma(p.top.r, u[2 * plane + rc + i], p.top.kx);
            gy[4] = -v[2 * plane + rc + i];
        }
    };
    // moment closure: f's needs the node's g as well
    auto close_f = [&]() {
        if (CLOSURE == 1 && (bottom || top)) {
            load_g();
            if (bottom) moment_closure_bottom<double, 0>(f, gx, gy, p.bot, p);
            if (top) moment_closure_top<double, 0>(f, gx, gy, p.top, p);
        }
    };
    auto close_g = [&]() {  // the g part of the same functions (their f results are not used)
        if (CLOSURE == 1) {
            double t[9] = {};
            if (bottom) moment_closure_bottom<double, 0>(t, gx, gy, p.bot, p);
            if (top) moment_closure_top<double, 0>(t, gx, gy, p.top, p);
        }
    };
    // population of slot k (f_k; 9 + a: g_x; 14 + a: g_y), also to the neighbouring band that pulls it
    auto put = [&](int k, double v) {
        if (!active) return;
        out[k * plane + rc + i] = v;
        const int a = k < 9 ? k : (k < 14 ? k - 9 : k - 14);
        const bool dn = a == 4 || a == 7 || a == 8, up = a == 2 || a == 5 || a == 6;
        const int o = (b ^ 1) * (19 * plane) + k * plane + i;
        if (dn && jl == 0 && band.below) band.below[o + (band.rows_below + 1) * nx] = v;
        if (up && jl == band.rows - 1 && band.above) band.above[o] = v;
    };

    if (role == 0) {
        load_f();
        close_f();
        const double s1 = f[1] + f[3], s2 = f[2] + f[4], s5 = f[5] + f[7], s6 = f[6] + f[8];
        const double drho = ((s1 + s2) + (s5 + s6)) + f[0];
        const double rho = 1.0 + drho;
        const double r = recip_seed(rho), e = ffma(-rho, r, 1.0), r3 = fmul(3.0, r);
        q[0] = drho;
        q[32] = ffma(r3, ffma(e, e, e), r3);
    } else if (role == 1) {
        load_f();
        close_f();
        const double d1 = f[1] - f[3], d5 = f[5] - f[7], d6 = f[6] - f[8];
        double jx = d1 + (d5 - d6);
        if (FORCE) jx = ffma(0.5, p.Fx, jx);
        q[64] = jx;
    } else if (role == 2) {
        load_f();
        close_f();
        const double d2 = f[2] - f[4], d5 = f[5] - f[7], d6 = f[6] - f[8];
        q[96] = d2 + (d5 + d6);
    } else {
        load_g();
        close_g();
        const double bx = ((gx[0] + gx[1]) + (gx[2] + gx[3])) + gx[4];
        const double dby = ((gy[0] + gy[1]) + (gy[2] + gy[3])) + gy[4];
        q[128] = bx;
        q[160] = dby;
        q[192] = p.B0 + dby;
    }
    asm volatile("bar.sync %0, 128;" ::"r"(quad + 1) : "memory");
    const double drho = q[0], inv3 = q[32], jx = q[64], jy = q[96], bx = q[128], dby = q[160], by = q[192];
    const double x3 = fmul(jx, inv3), y3 = fmul(jy, inv3);
    const double om1 = p.om1f;
    if (role == 3) {
        const double om1m = p.om1m;
        const double ce = fmul(p.owm1, ffma(x3, by, -fmul(y3, bx)));
        const double cb1 = fmul(p.owm1, bx), cd1 = fmul(p.owm1, dby);
        put(9, ffma(om1m, gx[0], fmul(p.owm0, bx)));
        put(10, ffma(om1m, gx[1], cb1));
        put(11, ffma(om1m, gx[2], cb1 - ce));
        put(12, ffma(om1m, gx[3], cb1));
        put(13, ffma(om1m, gx[4], cb1 + ce));
        put(14, ffma(om1m, gy[0], fmul(p.owm0, dby)));
        put(15, ffma(om1m, gy[1], cd1 + ce));
        put(16, ffma(om1m, gy[2], cd1));
        put(17, ffma(om1m, gy[3], cd1 - ce));
        put(18, ffma(om1m, gy[4], cd1));
        return;
    }
    const double xx = fmul(fmul(1.0 / 6.0, x3), x3), yy = fmul(fmul(1.0 / 6.0, y3), y3);
    double Q = fmul(p.ov, drho), kx = 0.0, Qx;
    if (FORCE) {
        kx = fmul(p.kv, x3);
        Q = ffma(-1.0 / 3.0, kx, Q);
        Qx = Q + kx;
    } else {
        Qx = Q;
    }
    const double P = p.ov + Q;
    if (role == 2) {
        const double h = xx + yy, xy = fmul(x3, y3);
        const double b5 = ffma(2.0, h, xy), b6 = ffma(2.0, h, -xy);
        const double omxy = fmul(fmul(p.cm, bx), by);
        double z = -omxy;
        if (FORCE) z = ffma(p.kv, y3, z);
        const double T5 = ffma(b5, P, Qx + z), T6 = ffma(b6, P, Qx - z);
        const double X = FORCE ? ffma(x3, P, p.kv) : fmul(x3, P), Y = fmul(y3, P);
        double O5 = X + Y, O8 = X - Y;
        if (FORCE) {
            O5 = ffma(p.kv, b5, O5);
            O8 = ffma(p.kv, b6, O8);
        }
        put(5, ffma(om1, f[5], T5 + O5));
        put(7, ffma(om1, f[7], T5 - O5));
        put(8, ffma(om1, f[8], T6 + O8));
        put(6, ffma(om1, f[6], T6 - O8));
        return;
    }
    const double P4 = fmul(4.0, P);
    const double om13 = fmul(p.cm, ffma(-bx, bx, fmul(dby, p.B0 + by)));
    if (role == 0) {
        const double b1 = ffma(2.0, xx, -yy);
        const double T1 = ffma(b1, P4, FORCE ? ffma(4.0, Qx, om13) : fmul(4.0, Q) + om13);
        const double X = FORCE ? ffma(x3, P, p.kv) : fmul(x3, P);
        const double O1 = FORCE ? ffma(p.kv, b1, X) : X;
        put(1, ffma(om1, f[1], ffma(4.0, O1, T1)));
        put(3, ffma(om1, f[3], ffma(-4.0, O1, T1)));
    } else {
        const double h = xx + yy, Q4 = fmul(4.0, Q), Y = fmul(y3, P);
        const double T2 = ffma(ffma(2.0, yy, -xx), P4, Q4 - om13), T0 = ffma(-h, P4, Q4);
        put(0, ffma(4.0, T0, fmul(om1, f[0])));
        put(2, ffma(om1, f[2], ffma(4.0, Y, T2)));
        put(4, ffma(om1, f[4], ffma(-4.0, Y, T2)));
    }
}

}  // namespace lks
