// Small kernels of one step, one warp (kinematics), one cluster (scalars), one thread (reset):
//  * kinematics: the insect frames at t^n (Sec. 3.1, 3.3; Eq. M_body_yawpitchroll),
//    in FP64, written as one Frame block read by every CTA of the physical pass;
//  * scalars: the deterministic final reduction of the physical pass's per-CTA
//    partial sums, the time step (Algorithm 1 step b), the integrating-factor
//    AB2 coefficients and exponential tables, and the force row
//    (Eqs. force_with_unst_corrections, moment_of_love);
//  * reset: the step state after a new initial condition.
#include <cooperative_groups.h>

#include "kernels.cuh"

#include "../../include/flusi.h"

namespace flusi {

namespace {

struct M3 {
    double a[9];
};

// A x
__device__ void apply(const M3& A, const double* x, double* y)
{
    double t0 = A.a[0] * x[0] + A.a[1] * x[1] + A.a[2] * x[2];
    double t1 = A.a[3] * x[0] + A.a[4] * x[1] + A.a[5] * x[2];
    double t2 = A.a[6] * x[0] + A.a[7] * x[1] + A.a[8] * x[2];
    y[0] = t0, y[1] = t1, y[2] = t2;
}

__device__ void cross3(const double* a, const double* b, double* c)
{
    double c0 = a[1] * b[2] - a[2] * b[1];
    double c1 = a[2] * b[0] - a[0] * b[2];
    double c2 = a[0] * b[1] - a[1] * b[0];
    c[0] = c0, c[1] = c1, c[2] = c2;
}

// Body-to-global matrix of the quaternion (e0, e1, e2, e3) as printed in
// Sec. 3.6; its transpose is the global-to-body matrix M_body.
__device__ M3 quat_to_global(const double* e)
{
    const double a = e[0], b = e[1], c = e[2], d = e[3];
    return {{a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c),
             2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b),
             2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d}};
}

// Free flight (Sec. 3.6, Eq. oh_my_god_look_a_vector): one AB2 step of the
// 13 body equations with the fluid step's dt and ratio r = dt/dt_prev (Euler
// when `first`).  State y = (x_cntr, u_cntr, quat, Omega_body); forcing: the
// row's total force and its total moment about x_cntr, taken into body axes.
__device__ void advance_body(flusi_insect* ins, StepState* st, const Frame& F, const double* row,
                             double dt, double r, int first)
{
    double Ft[3] = {0, 0, 0}, mg[3] = {0, 0, 0};
    for (int p = 0; p < 3; ++p)
        for (int i = 0; i < 3; ++i) {
            Ft[i] += row[2 + 6 * p + i];
            mg[i] += row[5 + 6 * p + i];
        }
    // a wing's moment is about its pivot: M_c = M_pivot + (pivot - x_cntr) x F
    for (int s = 0; s < 2 && s < ins->nwings; ++s) {
        const double arm[3] = {F.pv[s][0] - F.xc[0], F.pv[s][1] - F.xc[1], F.pv[s][2] - F.xc[2]};
        double c[3];
        cross3(arm, row + 2 + 6 * (1 + s), c);
        for (int i = 0; i < 3; ++i) mg[i] += c[i];
    }
    M3 Mb;
    for (int i = 0; i < 9; ++i) Mb.a[i] = F.Mb[i];
    double mb[3];
    apply(Mb, mg, mb);

    double y[13], f[13];
    const double* e = ins->quat;
    const double* W = ins->Omega_body;
    const double* J = ins->J_body;
    const double* dof = ins->dof;
    for (int i = 0; i < 3; ++i) {
        y[i] = ins->x_cntr[i];
        y[3 + i] = ins->u_cntr[i];
        y[10 + i] = W[i];
        f[i] = ins->u_cntr[i];
        f[3 + i] = dof[i] * Ft[i] / ins->mass;
    }
    f[5] -= dof[2] * ins->gravity;
    for (int i = 0; i < 4; ++i) y[6 + i] = e[i];
    // quaternion rate: half the product eps (x) (0, Omega^(b))
    f[6] = -0.5 * (e[1] * W[0] + e[2] * W[1] + e[3] * W[2]);
    f[7] = 0.5 * (e[0] * W[0] + e[2] * W[2] - e[3] * W[1]);
    f[8] = 0.5 * (e[0] * W[1] + e[3] * W[0] - e[1] * W[2]);
    f[9] = 0.5 * (e[0] * W[2] + e[1] * W[1] - e[2] * W[0]);
    // Euler's equations in principal body axes
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3, k = (i + 2) % 3;
        f[10 + i] = dof[3 + i] * ((J[j] - J[k]) * W[j] * W[k] + mb[i]) / J[i];
    }
    for (int i = 0; i < 13; ++i) {
        const double step = first ? f[i] : (1.0 + 0.5 * r) * f[i] - 0.5 * r * st->body_rhs_prev[i];
        y[i] += dt * step;
        st->body_rhs_prev[i] = f[i];
    }
    const double qn = sqrt(y[6] * y[6] + y[7] * y[7] + y[8] * y[8] + y[9] * y[9]);
    for (int i = 0; i < 3; ++i) {
        ins->x_cntr[i] = y[i];
        ins->u_cntr[i] = y[3 + i];
        ins->Omega_body[i] = y[10 + i];
    }
    for (int i = 0; i < 4; ++i) ins->quat[i] = y[6 + i] / qn;
}

}  // namespace

// ---- the frame block, by one warp.
//
// FP64 instructions cost the same with one lane active as with 32, and each
// waits for the one before it: on one thread the frame block was a chain of
// some two thousand of them (48 to 100 us a step, the longest kernel of a small
// grid).  Here every level of the computation is spread over lanes and handed
// on through shared memory: a harmonic per lane, an angle's sine and cosine per
// lane, an element of a matrix product per lane, a component of a rotated
// vector per lane, a corner of a bounding box per lane: 18 to 23 us.  A step of
// 48 x 36 x 24 went from 105 to 63 us with it; RK4 at 192^3, with contour wings
// and the later stages' frames beside the passes, from 1335 to 1044 us.
struct KinWork {
    flusi_insect I;
    Frame F;
    double harm[3][FLUSI_MAX_FOURIER][3];   // per angle and harmonic: value, first and second derivative
    double ang[3][3];                       // phi, alpha, theta and their derivatives
    double cs[8], sn[8];                    // psi, beta, gamma, eta_stroke, alpha, theta, phi, pi
    double Bx[9], By[9], Bz[9], B1[9];      // body rotations
    double Rt[9], Rpi[9], Ra[2][9], Rp[2][9], Ms[2][9], T[2][9], Mw[2][9];
    double vec[3][3];                       // angular velocities on their way to the global frame
    double rp[2][3], drp[2][3], in[2][3], din[2][3], v[2][3], dv[2][3];
    double lo[3], hi[3], rim, corner[3][8][3], arc[8][2];
};

// element e = 3 r + c of the rotation about an axis (rot_x, rot_y, rot_z)
__device__ double rot_elem(int axis, double c, double s, int e)
{
    const int r = e / 3, k = e - 3 * r;
    if (r == axis || k == axis) return r == k ? 1.0 : 0.0;
    if (r == k) return c;
    // the next axis in cyclic order carries +s
    return k == (r + 1) % 3 ? s : -s;
}
// element of A B, of A^T x and of A x
__device__ double mul_elem(const double* A, const double* B, int e)
{
    const int i = e / 3, j = e - 3 * i;
    return A[i * 3] * B[j] + A[i * 3 + 1] * B[3 + j] + A[i * 3 + 2] * B[6 + j];
}
__device__ double apply_t_elem(const double* A, const double* x, int i)
{
    return A[i] * x[0] + A[3 + i] * x[1] + A[6 + i] * x[2];
}
__device__ double apply_elem(const double* A, const double* x, int i)
{
    return A[3 * i] * x[0] + A[3 * i + 1] * x[1] + A[3 * i + 2] * x[2];
}
__device__ double cross_elem(const double* a, const double* b, int i)
{
    const int j = (i + 1) % 3, k = (i + 2) % 3;
    return a[j] * b[k] - a[k] * b[j];
}

// Body and wing orientations and angular velocities, pivots, and the parts'
// bounding boxes at time t, into w.F; h grows the boxes.  All 32 lanes call it.
__device__ void kinematics_frame(KinWork& w, double t, double h, int lane)
{
    const flusi_insect& I = w.I;
    Frame& F = w.F;
    const int trio = lane / 3, comp = lane - 3 * trio;     // lanes as triples of components
    const int nine = lane / 9, elem = lane - 9 * nine;     // lanes as matrices
    const bool flying = I.free_flight != 0;

    // ---- the angles' Fourier series and derivatives
    if (lane < 3 * FLUSI_MAX_FOURIER) {
        const int a = lane / FLUSI_MAX_FOURIER, i = lane - a * FLUSI_MAX_FOURIER;
        if (i < I.nfourier) {
            const double ca = a == 0 ? I.phi_a[i] : a == 1 ? I.alpha_a[i] : I.theta_a[i];
            const double cb = a == 0 ? I.phi_b[i] : a == 1 ? I.alpha_b[i] : I.theta_b[i];
            const double two_pi = 6.283185307179586476925286766559;
            const double om = two_pi * (i + 1) * I.freq;
            double sn, cs;
            sincos(om * t, &sn, &cs);
            const double c = ca * cs + cb * sn;
            w.harm[a][i][0] = c;
            w.harm[a][i][1] = om * (cb * cs - ca * sn);
            w.harm[a][i][2] = -(om * om * c);
        }
    }
    if (lane < 3) {
        F.xc[lane] = I.x_cntr[lane];
        F.uc[lane] = I.u_cntr[lane];
    }
    if (lane == 31) F.t = t;
    __syncwarp();
    if (lane < 9) {
        double acc = comp == 0 ? 0.5 * (trio == 0 ? I.phi_a0 : trio == 1 ? I.alpha_a0 : I.theta_a0) : 0.0;
        for (int i = 0; i < I.nfourier; ++i) acc += w.harm[trio][i][comp];
        w.ang[trio][comp] = acc;
    }
    __syncwarp();
    const double dphi = w.ang[0][1], dalpha = w.ang[1][1], dtheta = w.ang[2][1];

    // ---- sines and cosines, then the elementary rotations
    if (lane < 8) {
        const double pi = 3.141592653589793238462643383279;
        const double x = lane == 0 ? I.psi : lane == 1 ? I.beta : lane == 2 ? I.gamma : lane == 3 ? I.eta_stroke
                         : lane == 4 ? w.ang[1][0] : lane == 5 ? w.ang[2][0] : lane == 6 ? w.ang[0][0] : pi;
        sincos(x, &w.sn[lane], &w.cs[lane]);
    }
    __syncwarp();
    // the right wing mirrors the left: R_x(pi) in the stroke matrix and
    // (phi, alpha) -> (-phi, -alpha) in the wing matrix
    if (nine == 0) {
        w.Bx[elem] = rot_elem(0, w.cs[0], w.sn[0], elem);
        w.Ms[0][elem] = rot_elem(1, w.cs[3], w.sn[3], elem);
        w.Ra[0][elem] = rot_elem(1, w.cs[4], w.sn[4], elem);
        w.Rp[0][elem] = rot_elem(0, w.cs[6], w.sn[6], elem);
    } else if (nine == 1) {
        w.By[elem] = rot_elem(1, w.cs[1], w.sn[1], elem);
        w.Rpi[elem] = rot_elem(0, w.cs[7], w.sn[7], elem);
        w.Ra[1][elem] = rot_elem(1, w.cs[4], -w.sn[4], elem);
        w.Rp[1][elem] = rot_elem(0, w.cs[6], -w.sn[6], elem);
    } else if (nine == 2) {
        w.Bz[elem] = rot_elem(2, w.cs[2], w.sn[2], elem);
        w.Rt[elem] = rot_elem(2, w.cs[5], -w.sn[5], elem);
    }
    __syncwarp();
    // M_body = R_x R_y R_z (Sec. 3.1), or the quaternion's (Sec. 3.6)
    if (nine < 2) w.T[nine][elem] = mul_elem(w.Ra[nine], w.Rt, elem);
    else if (nine == 2) w.B1[elem] = mul_elem(w.Bx, w.By, elem);
    __syncwarp();
    if (nine < 2) {
        w.Mw[nine][elem] = mul_elem(w.T[nine], w.Rp[nine], elem);
    } else if (nine == 2) {
        double m = mul_elem(w.B1, w.Bz, elem);
        if (flying) {
            const M3 Q = quat_to_global(I.quat);
            const int at = 3 * (elem % 3) + elem / 3;   // its transpose
            for (int i = 0; i < 9; ++i)
                if (i == at) m = Q.a[i];
        }
        F.Mb[elem] = m;
    }
    if (nine == 0) w.Ms[1][elem] = mul_elem(w.Rpi, w.Ms[0], elem);
    __syncwarp();
    if (nine < 2) w.T[nine][elem] = mul_elem(w.Mw[nine], w.Ms[nine], elem);
    __syncwarp();
    if (nine < 2) F.Mw[nine][elem] = mul_elem(w.T[nine], F.Mb, elem);   // global -> wing frame

    // ---- angular velocities: triples 0, 1 the wings (stroke frame, then body,
    // then global), triple 2 the body (nested form of Sec. 3.1)
    if (lane < 9)
        w.vec[trio][comp] = trio < 2 ? (comp == 1 ? (trio == 0 ? dalpha : -dalpha) : 0.0) : (comp == 0 ? I.psi_dot : 0.0);
    __syncwarp();
    for (int k = 0; k < 5; ++k) {
        double y = 0.0;
        const bool on = lane < 9 && (trio < 2 || k < 3);
        if (on) {
            const double* A = trio == 2 ? (k == 0 ? w.Bx : k == 1 ? w.By : w.Bz)
                                        : (k == 0 ? w.Ra[trio] : k == 1 ? w.Rt : k == 2 ? w.Rp[trio] : k == 3 ? w.Ms[trio] : F.Mb);
            y = apply_t_elem(A, w.vec[trio], comp);
            if (trio < 2 && k == 0 && comp == 2) y += -dtheta;
            if (trio < 2 && k == 1 && comp == 0) y += trio == 0 ? dphi : -dphi;
            if (trio == 2 && k == 0 && comp == 1) y += I.beta_dot;
            if (trio == 2 && k == 1 && comp == 2) y += I.gamma_dot;
        }
        __syncwarp();
        if (on) w.vec[trio][comp] = y;
        __syncwarp();
    }
    if (lane < 6) F.Ow[trio][comp] = w.vec[trio][comp];
    else if (lane < 9) F.Ob[comp] = flying ? apply_t_elem(F.Mb, I.Omega_body, comp) : w.vec[2][comp];

    // In the wing frame Omega^(w) = e_a + Ra (e_t + Rt e_p) with
    // e_a = (0, alpha', 0), e_t = (0, 0, -theta'), e_p = (phi', 0, 0).  Both
    // factors are rotations about one fixed axis, so d/dt (Ra x) =
    // Ra x' - e_a x (Ra x) and d/dt (Rt x) = Rt x' - e_t x (Rt x).
    {
        const double sg = trio == 0 ? 1.0 : -1.0;
        const double ea[3] = {0, sg * dalpha, 0}, et[3] = {0, 0, -dtheta}, ep[3] = {sg * dphi, 0, 0};
        const double dea[3] = {0, sg * w.ang[1][2], 0}, det[3] = {0, 0, -w.ang[2][2]};
        const double dep[3] = {sg * w.ang[0][2], 0, 0};
        if (lane < 6) {
            w.rp[trio][comp] = apply_elem(w.Rt, ep, comp);
            w.drp[trio][comp] = apply_elem(w.Rt, dep, comp);
        }
        __syncwarp();
        if (lane < 6) {
            w.in[trio][comp] = (comp == 2 ? et[2] : 0.0) + w.rp[trio][comp];
            w.din[trio][comp] = (comp == 2 ? det[2] : 0.0) + w.drp[trio][comp] - cross_elem(et, w.rp[trio], comp);
        }
        __syncwarp();
        if (lane < 6) {
            w.v[trio][comp] = apply_elem(w.Ra[trio], w.in[trio], comp);
            w.dv[trio][comp] = apply_elem(w.Ra[trio], w.din[trio], comp);
        }
        __syncwarp();
        if (lane < 6) {
            F.Oww[trio][comp] = (comp == 1 ? ea[1] : 0.0) + w.v[trio][comp];
            F.dOww[trio][comp] = (comp == 1 ? dea[1] : 0.0) + w.dv[trio][comp] - cross_elem(ea, w.v[trio], comp);
            const double* pb = trio == 0 ? I.pivot_l : I.pivot_r;
            F.pv[trio][comp] = F.xc[comp] + apply_t_elem(F.Mb, pb, comp);
        }
    }

    // ---- bounding boxes (global) of the region where chi > 0
    // body-frame box of thorax, head and eyes; its corners, grown by h
    if (I.body_type == 3 && lane < 8) {
        // the arc x = x_c + r_c sin th, z = z_c + r_c cos th over
        // th0 -+ a/r_c: its ends and the quarter angles inside, grown by b
        const double rc = I.body_arc[0], xc = I.body_arc[1], zc = I.body_arc[2];
        const double th0 = atan2(-xc, -zc), t1 = th0 - I.body_a / rc, t2 = th0 + I.body_a / rc;
        const double half_pi = 1.5707963267948966192313216916398;
        const int k1 = (int)ceil(t1 / half_pi), k2 = (int)floor(t2 / half_pi);
        const int k = min(k1 - 1 + lane, k2 + 1);   // at most 4 quarter angles in an arc under a full turn
        const double th = k < k1 ? t1 : k > k2 ? t2 : k * half_pi;
        w.arc[lane][0] = xc + rc * sin(th);
        w.arc[lane][1] = zc + rc * cos(th);
    }
    double rim = 0.0;   // R(theta) <= a0/2 + sum sqrt(a_i^2 + b_i^2)
    if (I.wing_shape == 1) {
        if (lane < I.ncontour)
            rim = sqrt(I.contour_a[lane] * I.contour_a[lane] + I.contour_b[lane] * I.contour_b[lane]);
        for (int o = 16; o > 0; o >>= 1) rim += __shfl_xor_sync(0xffffffffu, rim, o);
        rim += 0.5 * I.contour_a0;
    }
    __syncwarp();
    if (lane < 3) {
        const double ey = I.body_type == 1 ? I.body_a : I.body_b;
        double lo = lane == 0 ? -I.body_a : -ey, hi = lane == 0 ? I.body_a : ey;
        if (I.body_type == 3 && lane != 1) {
            lo = 1e300;
            hi = -1e300;
            for (int k = 0; k < 8; ++k) {
                const double p = w.arc[k][lane == 0 ? 0 : 1];
                lo = fmin(lo, p - I.body_b);
                hi = fmax(hi, p + I.body_b);
            }
        }
        if (I.body_type >= 2 && I.head_r > 0) {
            lo = fmin(lo, I.head_x0[lane] - I.head_r);
            hi = fmax(hi, I.head_x0[lane] + I.head_r);
        }
        if (I.body_type >= 2 && I.eye_r > 0) {
            const double c = I.eye_x0[lane], m = lane == 1 ? -c : c;   // both eyes
            lo = fmin(lo, fmin(c, m) - I.eye_r);
            hi = fmax(hi, fmax(c, m) + I.eye_r);
        }
        w.lo[lane] = lo;
        w.hi[lane] = hi;
    }
    __syncwarp();
    if (lane < 24) {
        const int part = lane / 8, c = lane - 8 * part;
        double q[3];
        if (part == 0) {
            for (int i = 0; i < 3; ++i) q[i] = (c >> i) & 1 ? w.hi[i] + h : w.lo[i] - h;
        } else if (I.wing_shape == 1) {
            q[0] = c & 1 ? I.contour_xc + rim + h : I.contour_xc - rim - h;
            q[1] = c & 2 ? I.contour_yc + rim + h : I.contour_yc - rim - h;
            q[2] = c & 4 ? 0.5 * I.wing_h + h : -0.5 * I.wing_h - h;
        } else {
            q[0] = c & 1 ? I.wing_c_le + h : -I.wing_c_te - h;
            q[1] = c & 2 ? I.wing_R + h : -h;
            q[2] = c & 4 ? 0.5 * I.wing_h + h : -0.5 * I.wing_h - h;
        }
        const double* M = part == 0 ? F.Mb : F.Mw[part - 1];
        const double* at = part == 0 ? F.xc : F.pv[part - 1];
        for (int i = 0; i < 3; ++i) w.corner[part][c][i] = at[i] + apply_t_elem(M, q, i);
    }
    __syncwarp();
    if (lane < 18) {
        const int part = lane / 6, b = lane - 6 * part;
        const bool present = part == 0 ? I.body_type != 0 : part <= I.nwings;
        double v = b & 1 ? -1e300 : 1e300;
        if (present)
            for (int c = 0; c < 8; ++c) v = b & 1 ? fmax(v, w.corner[part][c][b / 2]) : fmin(v, w.corner[part][c][b / 2]);
        F.box[part][b] = v;
        if (b == 0) F.active[part] = present ? 1 : 0;
    } else if (lane == 18) {
        F.pad = 0;
    }
    __syncwarp();
}

// One warp: the FP64 frame block at the state's time (frac = 0) or at
// t0 + frac dt of the current step (the later RK4 stages, after k_scalars has
// written t0 and dt) and, with `with_t`, its FP32 and FP64 copies with the
// mask shape S (FrameT, at their offsets of the frame slot) for the x pass.
__global__ void __launch_bounds__(32)
k_kinematics(const flusi_insect* ins, const StepState* st, const StepCoef* coef, Frame* fr, double h, double frac,
             const Member* mb, const __grid_constant__ Shape S, int with_t, double inv_eta)
{
    __shared__ KinWork w;
    if (mb) {
        const Member& m = mb[blockIdx.z];
        ins = m.ins;
        st = m.st;
        coef = m.coef;
        fr = m.fr;
    }
    const int lane = threadIdx.x;
    static_assert(sizeof(flusi_insect) % 8 == 0 && sizeof(Frame) % 8 == 0, "word copies");
    for (int i = lane; i < (int)(sizeof(flusi_insect) / 8); i += 32)
        reinterpret_cast<double*>(&w.I)[i] = reinterpret_cast<const double*>(ins)[i];
    const double t = frac > 0.0 ? coef->t0 + frac * coef->dt : st->t;
    __syncwarp();
    kinematics_frame(w, t, h, lane);
    for (int i = lane; i < (int)(sizeof(Frame) / 8); i += 32)
        reinterpret_cast<double*>(fr)[i] = reinterpret_cast<const double*>(&w.F)[i];
    if (!with_t) return;
    frame_to_t<float>(const_cast<FrameT<float>*>(frame_t<float>(fr)), &w.F, &S, inv_eta, lane);
    frame_to_t<double>(const_cast<FrameT<double>*>(frame_t<double>(fr)), &w.F, &S, inv_eta, lane);
}

// A bounded wait on a barrier that nothing completes (the arrival count is 2
// and one thread arrives once): gives up after max_cycles and reports as the
// tile loads do.
__global__ void k_wait_probe(int* err, long long max_cycles)
{
    __shared__ unsigned long long bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 2);
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&bar)) : "memory");
    }
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0, max_cycles);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicCAS(err, 0, (int)FLUSI_ETIMEOUT);
}

__global__ void k_reset_state(StepState* st, StepCoef* coef)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    StepState s = {};
    *st = s;
    StepCoef c = {};
    *coef = c;
}

// A cluster of CTAs per solver.  Reduces part[nparts][kNumSums] in a fixed
// order, then forms the step's scalars.  `opts` = {cfl, dt_fixed, dt_max};
// dt_diff > 0 caps the adaptive step (the explicit-diffusion limit of RK4).
//
// FP64 arithmetic is a small fraction of FP32 here, and a warp instruction
// costs the FP64 units the same with one lane active as with 32: the work is
// spread over lanes (a slot and segment of the physical pass's CTAs per thread,
// a force or moment component per lane), and over the FP64 units of several
// SMs: every CTA of the cluster sums its share of the partials, takes the
// others' sums through distributed shared memory in rank order (so all hold the
// same totals and dt) and fills its share of the factor tables, rank 0 the force
// row meanwhile.  On one block it took 16 to 61 us, longer than the forward
// passes beside it wherever the physical pass has many small tiles.
constexpr int kScalarSeg = 6;   // segments of a CTA's share per slot: kNumSums * 6 = 240 threads
static_assert(kNumSums * kScalarSeg <= 256, "k_scalars runs 256 threads");

__global__ void __cluster_dims__(kScalarCtas, 1, 1) __launch_bounds__(256)
k_scalars(Geom g, const double* part, int nparts, StepState* st, StepCoef* coef, double* rows,
          int ring, double* etab, double3 opts, double dt_diff, const Frame* fr, flusi_insect* ins,
          const Member* mb)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    if (mb) {
        const Member& m = mb[blockIdx.z];
        part = m.part;
        st = m.st;
        coef = m.coef;
        rows = m.rows;
        etab = m.etab;
        fr = m.fr;
        ins = m.ins;
        g.nu = m.nu;
    }
    __shared__ double seg[kNumSums][kScalarSeg];
    __shared__ double own[kNumSums];
    __shared__ double tot[kNumSums];
    __shared__ double sh_dt;
    __shared__ int saw, any_saw;
    const int tid = threadIdx.x, T = blockDim.x;

    // every thread of the cluster reads the state before the first cluster
    // barrier; rank 0's thread 0 writes it only after that.  A block of a pass
    // beside this kernel may record a failure meanwhile: what each CTA's thread
    // 0 saw is exchanged with the sums, so that the cluster goes one way.
    const long long n = st->n;
    const double dt_prev = st->dt_prev;
    if (tid == 0) saw = *(volatile int*)&st->status;
    // slot k, segment s of this CTA: the partials of CTAs [s c, (s + 1) c) in
    // order; then the segments in order
    if (tid < kNumSums * kScalarSeg) {
        const int k = tid % kNumSums, sg = rank * kScalarSeg + tid / kNumSums;
        const int chunk = (nparts + kScalarCtas * kScalarSeg - 1) / (kScalarCtas * kScalarSeg);
        const int i0 = sg * chunk, i1 = min(nparts, i0 + chunk);
        const bool is_max = (k == kSumUmax2 || k == kSumBad);
        double acc = 0.0;
#pragma unroll 8
        for (int i = i0; i < i1; ++i) {
            const double v = part[(size_t)i * kNumSums + k];
            acc = is_max ? fmax(acc, v) : acc + v;
        }
        seg[k][tid / kNumSums] = acc;
    }
    __syncthreads();
    if (tid < kNumSums) {
        const bool is_max = (tid == kSumUmax2 || tid == kSumBad);
        double a = 0.0;
        for (int s2 = 0; s2 < kScalarSeg; ++s2) a = is_max ? fmax(a, seg[tid][s2]) : a + seg[tid][s2];
        own[tid] = a;
    }
    cluster.sync();
    if (tid < kNumSums) {
        const bool is_max = (tid == kSumUmax2 || tid == kSumBad);
        double a = 0.0;
        for (int r = 0; r < kScalarCtas; ++r) {
            const double v = cluster.map_shared_rank(own, r)[tid];
            a = is_max ? fmax(a, v) : a + v;
        }
        tot[tid] = a;
    } else if (tid == kNumSums) {
        int a = 0;
        for (int r = 0; r < kScalarCtas; ++r) a |= *cluster.map_shared_rank(&saw, r);
        any_saw = a;
    }
    __syncthreads();

    if (any_saw != 0 || tot[kSumBad] != 0.0) {
        if (rank == 0 && tid == 0) {
            if (any_saw == 0) atomicCAS(&st->status, 0, (int)FLUSI_ENONFINITE);
            coef->skip = 1;
        }
        cluster.sync();   // the others have read this CTA's sums
        return;
    }

    // time step (Algorithm 1 step b)
    const double umax = sqrt(tot[kSumUmax2]);
    if (tid == 0) {
        double dt;
        if (opts.y > 0.0) {
            dt = opts.y;
        } else {
            const double dmin = fmin(g.dx, fmin(g.dy, g.dz));
            dt = g.eta;
            if (umax > 0.0) dt = fmin(dt, opts.x * dmin / umax);
            if (opts.z > 0.0) dt = fmin(dt, opts.z);
            if (dt_diff > 0.0) dt = fmin(dt, dt_diff);
        }
        sh_dt = dt;
    }
    __syncthreads();
    const double dt = sh_dt;
    const int first = (n == 0);

    // integrating factors, separable per axis: E1 = e^{-nu |k|^2 dt},
    // E2 = e^{-nu |k|^2 (dt + dt_prev)}; layout [E1x Mx][E1y My][E1z Mz][E2x][E2y][E2z]
    // in FP64, then the same 2 Mt values rounded to FP32 (the FP32 update reads
    // those and converts nothing per mode)
    const double two_pi = 6.283185307179586476925286766559;
    const int Mt = g.Mx + g.My + g.Mz;
    float* etab32 = reinterpret_cast<float*>(etab + 2 * Mt);
    for (int i = (rank - 1) * T + tid; rank > 0 && i < 2 * Mt; i += (kScalarCtas - 1) * T) {
        int which = i / Mt, r = i % Mt;
        double k, tau = which == 0 ? dt : dt + dt_prev;
        if (r < g.Mx) k = two_pi * r / g.Lx;
        else if (r < g.Mx + g.My) k = two_pi * mode_of(r - g.Mx, g.Ky) / g.Ly;
        else k = two_pi * mode_of(r - g.Mx - g.My, g.Kz) / g.Lz;
        const double e = exp(-g.nu * k * k * tau);
        etab[i] = e;
        etab32[i] = float(e);
    }

    // force row: lane 3 p + i of rank 0's warp 0 takes component i of part p;
    // then the wing power (lanes 0, 1) and the rest (lane 0)
    if (rank == 0 && tid < 32) {
        double* row = rows + (size_t)(n % ring) * kRowCols;
        if (tid < 9) {
            const int p = tid / 3, i = tid % 3;
            const double dV = g.dx * g.dy * g.dz;
            const double* s = tot + 12 * p;
            double Fv = s[i] * dV / g.eta, Mv = s[3 + i] * dV / g.eta;
            const double Is = s[6 + i] * dV, Js = s[9 + i] * dV;
            if (!first) {
                const double inv_dtp = 1.0 / dt_prev;
                Fv += (Is - st->Is_prev[p][i]) * inv_dtp;
                Mv += (Js - st->Js_prev[p][i]) * inv_dtp;
            }
            row[2 + 6 * p + i] = Fv;
            row[5 + 6 * p + i] = Mv;
            st->Is_prev[p][i] = Is;
            st->Js_prev[p][i] = Js;
        }
        __syncwarp();
        const Frame& F = *fr;
        if (tid < 2) {   // wing power at t^n (Sec. 3.5, Eq. insect_power)
            const int s = tid;
            double pa = 0.0, pi = 0.0;
            if (s < ins->nwings) {
                const double* m = row + 5 + 6 * (1 + s);
                pa = -(m[0] * F.Ow[s][0] + m[1] * F.Ow[s][1] + m[2] * F.Ow[s][2]);
                const double* J = ins->J_wing;   // xx yy zz xy xz yz
                const M3 Jm = {{J[0], J[3], J[4], J[3], J[1], J[5], J[4], J[5], J[2]}};
                const double* w = F.Oww[s];
                double Jw[3], Jdw[3], c[3];
                apply(Jm, w, Jw);
                apply(Jm, F.dOww[s], Jdw);
                cross3(w, Jw, c);
                pi = w[0] * (Jdw[0] + c[0]) + w[1] * (Jdw[1] + c[1]) + w[2] * (Jdw[2] + c[2]);
            }
            row[22 + s] = pa;
            row[24 + s] = pi;
        }
        __syncwarp();
        if (tid == 0) {
            StepCoef c;
            c.dt = dt;
            c.n = n;
            c.first = first;
            c.t0 = st->t;
            c.skip = 0;
            if (first) {
                c.c_now = dt;
                c.c_old = 0.0;
            } else {
                double r = dt / dt_prev;
                c.c_now = dt * (1.0 + 0.5 * r);
                c.c_old = dt * 0.5 * r;
            }
            *coef = c;
            row[0] = st->t;
            row[1] = dt;
            row[20] = 0.5 * tot[kSumEkin] * g.dx * g.dy * g.dz;
            row[21] = umax;

            if (ins->free_flight) advance_body(ins, st, F, row, dt, first ? 0.0 : dt / dt_prev, first);

            st->t += dt;
            st->dt_prev = dt;
            st->n = n + 1;
        }
    }
    cluster.sync();   // every CTA has read the others' sums
}

}  // namespace flusi
