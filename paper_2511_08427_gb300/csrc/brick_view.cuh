// Per-(brick, view) constants of the output-stationary matched adjoints (FP64 on the device), shared by the
// 3D bricks (k_adjoint_brick.cu) and the 2D ones (k_adjoint2d.cu).
#pragma once

#include "device_common.cuh"

namespace pyronn {

struct BrickView {
    int u_lo, v_lo, nu_r, nv_r;     // footprint rectangle (nu_r == 0: empty)
    float A[3];                     // corner-ray point on the brick plane, relative to the brick centre
    float Eu[3], Ev[3];             // per-pixel steps of that point
    float D[3];                     // corner-ray direction (unnormalised)
    float Cu[3], Cv[3];             // per-pixel steps of the direction (zero for parallel beams)
    float inv_nD, nD2;              // 1 / |D|, |D|^2
    float dref[3];                  // D / |D|
    float f;                        // phase: (X_b - C) . dref = (K + f) dt, 0 <= f < 1
    int pad;
};

// Detector position of a point X relative to the volume centre; false behind the source plane
static __device__ __forceinline__ bool brick_corner(const OpParams &p, const double *x, const double X[3], double &u, double &v) {
    if (p.perspective) {
        double a = x[0] * X[0] + x[1] * X[1] + x[2] * X[2] + x[3];
        double b = x[4] * X[0] + x[5] * X[1] + x[6] * X[2] + x[7];
        double w = x[8] * X[0] + x[9] * X[1] + x[10] * X[2] + x[11];
        if (!(w > 0.0)) return false;
        u = a / w;
        v = b / w;
    } else {
        double Y[3] = {X[0] - x[0], X[1] - x[1], X[2] - x[2]};
        u = ((Y[0] * x[3] + Y[1] * x[4] + Y[2] * x[5]) - p.ou) / p.du + 0.5 * (p.det.nu - 1);
        v = ((Y[0] * x[6] + Y[1] * x[7] + Y[2] * x[8]) - p.ov) / p.dv + 0.5 * (p.det.nv - 1);
    }
    return true;
}

// FP64 per-(brick, view) set-up for a footprint with the corner (u_lo, v_lo). Xb: brick centre relative to the volume
// centre (world mm). at (2D): A[0], A[1], Eu[0], Eu[1] unrounded.
static __device__ void brick_view_rays(const OpParams &p, int view, const double Xb[3], int u_lo, int v_lo, BrickView &bv,
                                       double *at = nullptr) {
    const double *x = p.views64 + (size_t)view * VIEW64_STRIDE;
    const double hu = 0.5 * (p.det.nu - 1), hv = 0.5 * (p.det.nv - 1);
    double A[3], Eu[3], Ev[3], D[3], Cu[3], Cv[3];
    if (p.perspective) {
        const double *S = x + 12, *c0 = x + 15, *c1 = x + 18, *c2 = x + 21, *nrm = x + 24;
        double den = x[27];
        double lam = ((Xb[0] - S[0]) * nrm[0] + (Xb[1] - S[1]) * nrm[1] + (Xb[2] - S[2]) * nrm[2]) / den;
        for (int i = 0; i < 3; ++i) {
            D[i] = c2[i] + u_lo * c0[i] + v_lo * c1[i];
            A[i] = S[i] + lam * D[i] - Xb[i];
            Eu[i] = lam * c0[i];
            Ev[i] = lam * c1[i];
            Cu[i] = c0[i];
            Cv[i] = c1[i];
        }
    } else {
        const double *Dc = x, *eu = x + 3, *ev = x + 6, *d = x + 9;
        double su = (u_lo - hu) * p.du + p.ou, sv = (v_lo - hv) * p.dv + p.ov;
        double a0[3], du_[3], dv_[3];
        for (int i = 0; i < 3; ++i) {
            a0[i] = Dc[i] + su * eu[i] + sv * ev[i] - Xb[i];   // corner-ray origin relative to X_b
            du_[i] = p.du * eu[i];
            dv_[i] = p.dv * ev[i];
        }
        double pa = a0[0] * d[0] + a0[1] * d[1] + a0[2] * d[2];
        double pu = du_[0] * d[0] + du_[1] * d[1] + du_[2] * d[2];
        double pv = dv_[0] * d[0] + dv_[1] * d[1] + dv_[2] * d[2];
        for (int i = 0; i < 3; ++i) {
            A[i] = a0[i] - pa * d[i];
            Eu[i] = du_[i] - pu * d[i];
            Ev[i] = dv_[i] - pv * d[i];
            D[i] = d[i];
            Cu[i] = 0.0;
            Cv[i] = 0.0;
        }
    }
    double nD2 = D[0] * D[0] + D[1] * D[1] + D[2] * D[2];
    double nD = sqrt(nD2);
    double dref[3] = {D[0] / nD, D[1] / nD, D[2] / nD};
    double T = (Xb[0] * dref[0] + Xb[1] * dref[1] + Xb[2] * dref[2]) / (double)p.dt;
    double K = floor(T);
    for (int i = 0; i < 3; ++i) {
        bv.A[i] = (float)A[i]; bv.Eu[i] = (float)Eu[i]; bv.Ev[i] = (float)Ev[i];
        bv.D[i] = (float)D[i]; bv.Cu[i] = (float)Cu[i]; bv.Cv[i] = (float)Cv[i];
        bv.dref[i] = (float)dref[i];
    }
    if (at) at[0] = A[0], at[1] = A[1], at[2] = Eu[0], at[3] = Eu[1];
    bv.inv_nD = (float)(1.0 / nD);
    bv.nD2 = (float)nD2;
    bv.f = (float)(T - K);
}

// FP64 per-(brick, view) set-up. Xb: brick centre relative to the volume centre (world mm);
// ext_lo / ext_hi: the extended brick (one voxel around it) relative to the volume centre.
static __device__ void brick_view_setup(const OpParams &p, int view, const double Xb[3], const double ext_lo[3],
                                 const double ext_hi[3], BrickView &bv) {
    const double *x = p.views64 + (size_t)view * VIEW64_STRIDE;
    const int nu = p.det.nu, nv = p.det.nv;
    // footprint: project the eight corners of the extended brick
    double umin = 1e300, umax = -1e300, vmin = 1e300, vmax = -1e300;
    bool behind = false;
    for (int c = 0; c < 8; ++c) {
        double X[3] = {(c & 1) ? ext_hi[0] : ext_lo[0], (c & 2) ? ext_hi[1] : ext_lo[1],
                       (c & 4) ? ext_hi[2] : ext_lo[2]};
        double u, v;
        if (!brick_corner(p, x, X, u, v)) {
            behind = true;
            continue;
        }
        umin = fmin(umin, u); umax = fmax(umax, u);
        vmin = fmin(vmin, v); vmax = fmax(vmax, v);
    }
    int u_lo, u_hi, v_lo, v_hi;
    if (behind) {
        u_lo = 0; u_hi = nu - 1; v_lo = 0; v_hi = nv - 1;
    } else {
        umin = fmax(umin, -2.0); umax = fmin(umax, (double)nu + 1.0);
        vmin = fmax(vmin, -2.0); vmax = fmin(vmax, (double)nv + 1.0);
        u_lo = max((int)ceil(umin) - 1, 0); u_hi = min((int)floor(umax) + 1, nu - 1);
        v_lo = max((int)ceil(vmin) - 1, 0); v_hi = min((int)floor(vmax) + 1, nv - 1);
    }
    bv.u_lo = u_lo; bv.v_lo = v_lo;
    bv.nu_r = (u_hi >= u_lo && v_hi >= v_lo) ? u_hi - u_lo + 1 : 0;
    bv.nv_r = (u_hi >= u_lo && v_hi >= v_lo) ? v_hi - v_lo + 1 : 0;
    if (bv.nu_r == 0) return;

    brick_view_rays(p, view, Xb, u_lo, v_lo, bv);
}

}  // namespace pyronn
