// Physical-space pieces of the x pass shared by its kernels: the FP64 frame
// block turned into the pass's precision, the signed distances of the
// insect's parts and the smoothed mask (Sec. 3, Eq.
// smoothing_mask_as_function_of_delta), the solid velocity (Eqs.
// body_velocity_field, wing_velocity_field), and the pre- and
// post-processing that turns a length-nx real transform into a length-nx/2
// complex one.
#pragma once

#include "kernels.cuh"

namespace flusi {
namespace {

// The block's copy of the frame in T (written by the kinematics kernel),
// by every thread of the block in 4-byte words.
template <typename T> __device__ __forceinline__ void load_frame_t(FrameT<T>* dst, const Frame* fr)
{
    static_assert(sizeof(FrameT<T>) % 4 == 0, "word copy");
    const unsigned* src = reinterpret_cast<const unsigned*>(frame_t<T>(fr));
    unsigned* d = reinterpret_cast<unsigned*>(dst);
    for (int i = threadIdx.x; i < (int)(sizeof(FrameT<T>) / 4); i += blockDim.x) d[i] = src[i];
}

// The pass's copy of the frame (FP64 on the device) and mask shape in T.
template <typename T>
__device__ void setup_frame(FrameT<T>& f, const Frame& F, const Shape& S, double inv_eta)
{
    for (int i = 0; i < 3; ++i) {
        f.xc[i] = T(F.xc[i]);
        f.uc[i] = T(F.uc[i]);
        f.Ob[i] = T(F.Ob[i]);
        f.active[i] = F.active[i];
        for (int s2 = 0; s2 < 2; ++s2) {
            f.pv[s2][i] = T(F.pv[s2][i]);
            f.Ow[s2][i] = T(F.Ow[s2][i]);
        }
        for (int k = 0; k < 6; ++k) f.box[i][k] = T(F.box[i][k]);
        f.head_x0[i] = T(S.head_x0[i]);
        f.eye_x0[i] = T(S.eye_x0[i]);
    }
    for (int i = 0; i < 9; ++i) {
        f.Mb[i] = T(F.Mb[i]);
        f.Mw[0][i] = T(F.Mw[0][i]);
        f.Mw[1][i] = T(F.Mw[1][i]);
    }
    f.h = T(S.h);
    f.a = T(S.body_a);
    f.b = T(S.body_b);
    f.c_le = T(S.c_le);
    f.c_te = T(S.c_te);
    f.R = T(S.R);
    f.ht = T(S.ht);
    f.inv_eta = T(inv_eta);
    f.body_type = S.body_type;
    f.profile = S.profile;
    f.wing_shape = S.wing_shape;
    f.ncontour = S.ncontour;
    f.head_r = T(S.head_r);
    f.eye_r = T(S.eye_r);
    f.cxc = T(S.contour_xc);
    f.cyc = T(S.contour_yc);
    f.ca0 = T(S.contour_a0);
    for (int i = 0; i < FLUSI_MAX_CONTOUR; ++i) {
        f.ca[i] = T(S.contour_a[i]);
        f.cb[i] = T(S.contour_b[i]);
    }
    f.arc_r = T(S.arc_r);
    f.arc_x = T(S.arc_x);
    f.arc_z = T(S.arc_z);
    f.arc_ux = T(S.arc_ux);
    f.arc_uz = T(S.arc_uz);
    for (int e = 0; e < 2; ++e) {
        f.arc_end[e][0] = T(S.arc_end[e][0]);
        f.arc_end[e][1] = T(S.arc_end[e][1]);
    }
    if (S.body_type == 0) f.active[0] = 0;
    if (S.nwings < 1) f.active[1] = 0;
    if (S.nwings < 2) f.active[2] = 0;
}

// Signed distance of the body in its frame (Sec. 3.2): thorax (sphere,
// ellipsoid, or the ellipsoid bent along a circular arc as for the fruit fly
// of Sec. 5.3), joined with the head and eye spheres by the minimum.
template <typename T>
__device__ __forceinline__ T body_delta(const FrameT<T>& F, const T* xb)
{
    T delta;
    if (F.body_type == 1) {
        delta = sqrt(xb[0] * xb[0] + xb[1] * xb[1] + xb[2] * xb[2]) - F.a;
    } else {
        if (F.body_type == 3) {
            // arc length s of the point's angle about the circle's centre,
            // from the direction u towards the body origin; the offset from
            // the centre line in the circle's plane is r - r_c, across it y
            const T vx = xb[0] - F.arc_x, vz = xb[2] - F.arc_z;
            const T s = F.arc_r * atan2(vx * F.arc_uz - vz * F.arc_ux, vx * F.arc_ux + vz * F.arc_uz);
            if (fabs(s) <= F.a) {
                const T dr = sqrt(vx * vx + vz * vz) - F.arc_r, q = s / F.a;
                delta = sqrt(dr * dr + xb[1] * xb[1]) - F.b * sqrt(fmax(T(0), T(1) - q * q));
            } else {
                const T* e = F.arc_end[s > T(0) ? 1 : 0];
                const T ex = xb[0] - e[0], ez = xb[2] - e[1];
                delta = sqrt(ex * ex + xb[1] * xb[1] + ez * ez);
            }
        } else {
            T rr = sqrt(xb[1] * xb[1] + xb[2] * xb[2]), ax = fabs(xb[0]);
            if (ax <= F.a) {
                T q = xb[0] / F.a;
                delta = rr - F.b * sqrt(fmax(T(0), T(1) - q * q));
            } else {
                delta = sqrt(rr * rr + (ax - F.a) * (ax - F.a));
            }
        }
        if (F.head_r > T(0)) {
            const T e0 = xb[0] - F.head_x0[0], e1 = xb[1] - F.head_x0[1], e2 = xb[2] - F.head_x0[2];
            delta = fmin(delta, sqrt(e0 * e0 + e1 * e1 + e2 * e2) - F.head_r);
        }
        if (F.eye_r > T(0)) {
            for (int s = 0; s < 2; ++s) {
                const T y0 = s == 0 ? F.eye_x0[1] : -F.eye_x0[1];
                const T e0 = xb[0] - F.eye_x0[0], e1 = xb[1] - y0, e2 = xb[2] - F.eye_x0[2];
                delta = fmin(delta, sqrt(e0 * e0 + e1 * e1 + e2 * e2) - F.eye_r);
            }
        }
    }
    return delta;
}

// Signed distance of a wing in its frame (Sec. 3.4): the rectangular plate,
// or the contour R(theta) = a0/2 + sum a_i cos(i theta) + b_i sin(i theta)
// with cos, sin of i theta from the angle-addition recurrence.
template <typename T>
__device__ __forceinline__ T wing_delta(const FrameT<T>& F, const T* xw)
{
    const T dz = fabs(xw[2]) - T(0.5) * F.ht;
    if (F.wing_shape == 1) {
        const T dx = xw[0] - F.cxc, dy = xw[1] - F.cyc;
        const T r = sqrt(dx * dx + dy * dy);
        const T c1 = r > T(0) ? dx / r : T(1), s1 = r > T(0) ? dy / r : T(0);
        T R = T(0.5) * F.ca0, ci = c1, si = s1;
        for (int i = 0; i < F.ncontour; ++i) {
            R += F.ca[i] * ci + F.cb[i] * si;
            const T cn = ci * c1 - si * s1;
            si = si * c1 + ci * s1;
            ci = cn;
        }
        return fmax(dz, r - R);
    }
    return fmax(fmax(xw[0] - F.c_le, -xw[0] - F.c_te), fmax(fmax(xw[1] - F.R, -xw[1]), dz));
}

template <typename T> __device__ __forceinline__ T profile_chi(int profile, T d, T h)
{
    if (profile == 1) return T(0.5) * (T(1) - tanh(d / h));
    if (d <= -h) return T(1);
    if (d >= h) return T(0);
    return T(0.5) * (T(1) + cospi((d + h) / (T(2) * h)));
}

template <typename T>
__device__ __forceinline__ void cross3(const T* a, const T* b, T* c)
{
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}

// u x w of two points at once (packed pairs), rounded as cross3 rounds it
__device__ __forceinline__ void cross3_pair(const float2* u, const float2* w, float2* c)
{
    const float2 minus = make_float2(-1.0f, -1.0f);
    const float2 v[3] = {__fmul2_rn(w[0], minus), __fmul2_rn(w[1], minus), __fmul2_rn(w[2], minus)};
    c[0] = __ffma2_rn(u[1], w[2], __fmul2_rn(u[2], v[1]));
    c[1] = __ffma2_rn(u[2], w[0], __fmul2_rn(u[0], v[2]));
    c[2] = __ffma2_rn(u[0], w[1], __fmul2_rn(u[1], v[0]));
}

// Mask, colour (0 fluid, 1 body, 2/3 wings) and solid velocity at X.
template <typename T>
__device__ __forceinline__ void solid_at(const FrameT<T>& F, const T* X, const bool* inrow, T& chi,
                                         int& col, T* us)
{
    chi = T(0);
    col = 0;
    us[0] = us[1] = us[2] = T(0);
    if (!(inrow[0] | inrow[1] | inrow[2])) return;
    T d[3] = {X[0] - F.xc[0], X[1] - F.xc[1], X[2] - F.xc[2]};
    if (inrow[0] && X[0] >= F.box[0][0] && X[0] <= F.box[0][1]) {
        T xb[3];
        for (int i = 0; i < 3; ++i) xb[i] = F.Mb[3 * i] * d[0] + F.Mb[3 * i + 1] * d[1] + F.Mb[3 * i + 2] * d[2];
        const T delta = body_delta(F, xb);
        T c = profile_chi(F.profile, delta, F.h);
        if (c > chi) {
            chi = c;
            col = 1;
            T w[3];
            cross3(F.Ob, d, w);
            for (int i = 0; i < 3; ++i) us[i] = F.uc[i] + w[i];
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if (!(inrow[1 + s] && X[0] >= F.box[1 + s][0] && X[0] <= F.box[1 + s][1])) continue;
        const T* M = F.Mw[s];
        T e[3] = {X[0] - F.pv[s][0], X[1] - F.pv[s][1], X[2] - F.pv[s][2]};
        T xw[3];
        for (int i = 0; i < 3; ++i) xw[i] = M[3 * i] * e[0] + M[3 * i + 1] * e[1] + M[3 * i + 2] * e[2];
        const T delta = wing_delta(F, xw);
        T c = profile_chi(F.profile, delta, F.h);
        if (c > chi) {
            chi = c;
            col = 2 + s;
            T w[3], v[3];
            cross3(F.Ob, d, w);
            cross3(F.Ow[s], e, v);
            for (int i = 0; i < 3; ++i) us[i] = F.uc[i] + w[i] + v[i];
        }
    }
}

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}


// a b + c, rounded once
__device__ __forceinline__ float fmadd(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmadd(double a, double b, double c) { return __fma_rn(a, b, c); }

// a + b rounded, and in e what the rounding dropped (two-sum; Knuth, TAOCP 4.2.2)
__device__ __forceinline__ float two_sum(float a, float b, float& e)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}
__device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2& e)
{
    const float2 s = cadd(a, b), t = csub(s, a);
    e = cadd(csub(a, csub(s, t)), csub(b, t));
    return s;
}
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return cadd(a, b); }
// h + l + m += x + y + z, three parts of falling size (V: float, or two sums packed);
// only the last part is rounded, some 70 bits below the first
template <class V> __device__ __forceinline__ void triple_add(V& h, V& l, V& m, V x, V y, V z)
{
    V e1, e2, e3;
    h = two_sum(h, x, e1);
    l = two_sum(l, y, e2);
    l = two_sum(l, e1, e3);
    m = add(add(m, z), add(e2, e3));
}
__device__ __forceinline__ float lane_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float2 lane_xor(float2 v, int o) { return make_float2(lane_xor(v.x, o), lane_xor(v.y, o)); }

// The warp totals of 12 per-lane values in FP64, added into w[0..11]: a
// reduce-scatter over 16 slots (12 values, 4 zeros), halving the slots per lane at
// each of the xor-16, 8, 4, 2 exchanges, then one xor-1 add; lane 2i + 1 (bits 4..1
// = i) ends with the total of slot i.  Every lane of the warp calls it.
__device__ __forceinline__ void warp_sums12(const double* v, double* w, int lane)
{
    double d[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) d[k] = k < 12 ? v[k] : 0.0;
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = (lane & (2 * h)) != 0;   // this lane keeps the upper half
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double keep = up ? d[k + h] : d[k];
            const double send = up ? d[k] : d[k + h];
            d[k] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
        }
    }
    d[0] += __shfl_xor_sync(0xffffffffu, d[0], 1);
    const int slot = (lane >> 1) & 15;
    if ((lane & 1) && slot < 12) w[slot] += d[0];
}

// The same for FP32 values, with no more error: FP64 issues one warp instruction in
// some 17 cycles of an SM, and with FP64 sums (12 conversions and 16 adds per warp)
// they, not the line transforms, set the time of tiles with penalized points.  The
// tree therefore runs in FP32 instructions on values of three parts, of which only
// what lies some 70 bits below the largest is ever rounded; FP64 adds the parts and
// everything above the warp.  x pass with a sphere of 0.3 box lengths at 256^3: FP64
// tree 286 us, this one 244 (156 without a body; with two parts, 48 bits, 232).  Sums
// kept per lane over a tile cost registers that the transforms need: 512^3 x pass
// 1090 -> 1171 us.  Where a partial sum could leave the FP32 range, and
// for infinities, the warp takes the FP64 tree.
__device__ __forceinline__ void warp_sums12(const float* v, double* w, int lane)
{
    float big[4];   // (a NaN is passed over here: it comes out as one either way)
#pragma unroll
    for (int k = 0; k < 4; ++k) big[k] = fmaxf(fmaxf(fabsf(v[3 * k]), fabsf(v[3 * k + 1])), fabsf(v[3 * k + 2]));
    if (__any_sync(0xffffffffu, fmaxf(fmaxf(fmaxf(big[0], big[1]), big[2]), big[3]) >= 0x1p120f)) {   // 32 lanes of less stay under 2^125
        double d[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) d[k] = double(v[k]);
        warp_sums12(d, w, lane);
        return;
    }
    // pairs of neighbouring slots
    float2 h[4], l[4], m[2];
    const bool up16 = (lane & 16) != 0;   // this lane keeps the upper half
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 low = make_float2(v[2 * k], v[2 * k + 1]);
        const float2 top = k < 2 ? make_float2(v[2 * k + 8], v[2 * k + 9]) : make_float2(0.0f, 0.0f);
        h[k] = two_sum(up16 ? top : low, lane_xor(up16 ? low : top, 16), l[k]);   // two parts hold it
    }
#pragma unroll
    for (int n = 2; n >= 1; n >>= 1) {
        const bool up = (lane & (4 * n)) != 0;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            if (n == 2) m[k] = make_float2(0.0f, 0.0f);
            const float2 x = lane_xor(up ? h[k] : h[k + n], 4 * n), y = lane_xor(up ? l[k] : l[k + n], 4 * n);
            const float2 z = n == 2 ? make_float2(0.0f, 0.0f) : lane_xor(up ? m[0] : m[1], 4);
            h[k] = up ? h[k + n] : h[k];
            l[k] = up ? l[k + n] : l[k];
            if (n == 1) m[0] = up ? m[1] : m[0];
            triple_add(h[k], l[k], m[k], x, y, z);
        }
    }
    const bool up = (lane & 2) != 0;
    const float x = lane_xor(up ? h[0].x : h[0].y, 2), y = lane_xor(up ? l[0].x : l[0].y, 2),
                z = lane_xor(up ? m[0].x : m[0].y, 2);
    float a = up ? h[0].y : h[0].x, b = up ? l[0].y : l[0].x, c = up ? m[0].y : m[0].x;
    triple_add(a, b, c, x, y, z);
    const float x1 = lane_xor(a, 1), y1 = lane_xor(b, 1), z1 = lane_xor(c, 1);
    triple_add(a, b, c, x1, y1, z1);
    const int slot = (lane >> 1) & 15;
    if ((lane & 1) && slot < 12) w[slot] += double(a) + (double(b) + double(c));
}

// c2r pre-processing: Z[k] = (X[k] + X*[m]) + i (X[k] - X*[m]) w^{-k} with the
// mirror value Xm = X[nh - k].
template <typename T>
__device__ __forceinline__ cplx<T> c2r_pre(cplx<T> Xk, cplx<T> Xm, cplx<T> wk)
{
    // s + i d conj(w) with s = Xk + conj(Xm), d = Xk - conj(Xm), as fused
    // multiply-adds: (s.x - d.y w.x + d.x w.y, s.y + d.x w.x + d.y w.y)
    const T sx = Xk.x + Xm.x, sy = Xk.y - Xm.y, dx = Xk.x - Xm.x, dy = Xk.y + Xm.y;
    return mkc<T>(fmadd(dx, wk.y, fmadd(-dy, wk.x, sx)), fmadd(dy, wk.y, fmadd(dx, wk.x, sy)));
}

// r2c post-processing: X[k] = E + w^k O, E = (Z[k] + Z*[m])/2, O = -i (Z[k] - Z*[m])/2.
template <typename T>
__device__ __forceinline__ cplx<T> r2c_post(cplx<T> Zk, cplx<T> Zm, cplx<T> wk)
{
    // with a = Zk + conj(Zm), b = Zk - conj(Zm): E + w O = (a + w (-i b)) / 2
    // = (a.x + w.x b.y + w.y b.x, a.y + w.y b.y - w.x b.x) / 2, as fused
    // multiply-adds (the halving is exact)
    const T ax = Zk.x + Zm.x, ay = Zk.y - Zm.y, bx = Zk.x - Zm.x, by = Zk.y + Zm.y;
    return mkc<T>(T(0.5) * fmadd(wk.y, bx, fmadd(wk.x, by, ax)), T(0.5) * fmadd(-wk.x, bx, fmadd(wk.y, by, ay)));
}

// c2r pre-processing with X[nh - k] = 0 (a mode that the 2/3 rule drops): the
// same value as c2r_pre(Xk, 0, wk) in half the operations.
template <typename T>
__device__ __forceinline__ cplx<T> c2r_pre_nomirror(cplx<T> Xk, cplx<T> wk)
{
    return mkc<T>(fmadd(Xk.x, wk.y, fmadd(-Xk.y, wk.x, Xk.x)), fmadd(Xk.y, wk.y, fmadd(Xk.x, wk.x, Xk.y)));
}
// ... and with X[k] = 0.
template <typename T>
__device__ __forceinline__ cplx<T> c2r_pre_dropped(cplx<T> Xm, cplx<T> wk)
{
    return mkc<T>(fmadd(-Xm.x, wk.y, fmadd(-Xm.y, wk.x, Xm.x)), fmadd(Xm.y, wk.y, fmadd(-Xm.x, wk.x, -Xm.y)));
}

// Registers t of a lane's line elements k = j + L t, t < R = nh / L, that can
// hold a mode kept by the 2/3 rule (k <= nx/3 = 2 nh / 3); the others are zero.
template <int R, int L> constexpr int sq_kept() { return (2 * R * L / 3) / L + 1; }
// Registers t whose element is a kept mode on every lane, under the strict rule
// (nx/3 - 1 where 3 divides nx) too: they are loaded and stored without a test.
template <int R, int L> constexpr int sq_always()
{
    const int n = 2 * R * L, modes = (n % 3 == 0 ? n / 3 - 1 : n / 3) + 1;
    return modes / L;
}

template <typename T, int R, int L>
__device__ __forceinline__ void sq_exchange_pre(cplx<T>* x, int j, const cplx<T>* twx)
{
    // x[t] holds X[j + L t]; on return x[t] = Z[j + L t] (c2r pre-processing).
    // The mirror nh - k of k = j + L t is element R-1-t of lane L-j for j != 0,
    // and lane 0's own element R-t (t = 0: X[nh], a dropped mode, zero).  One
    // branch-free loop serves both: lane 0 "sends itself" elements s+1 and R-s
    // where the other lanes send elements s and R-1-s.  The pairs (s, R-1-s)
    // go from the middle outwards, so every element read is still unmodified
    // (element s+1 was overwritten the iteration before: carried from there).
    // Elements t >= NT hold dropped modes on every lane: nothing is exchanged
    // for them.
    constexpr int NT = sq_kept<R, L>();
    const int partner = (L - j) & (L - 1);
    const bool self = j == 0;
    cplx<T> carry = x[R / 2];   // the original element s + 1
#pragma unroll
    for (int s = R / 2 - 1; s >= 0; --s) {
        const cplx<T> xs = x[s], xt = x[R - 1 - s];
        const cplx<T> sa = self ? carry : xs;   // mirror of element R-1-s
        cplx<T> a, b;
        a.x = __shfl_sync(0xffffffffu, sa.x, partner, L);
        a.y = __shfl_sync(0xffffffffu, sa.y, partner, L);
        if (R - 1 - s < NT) {
            const cplx<T> up = s == 0 ? mkc<T>(0, 0) : x[s == 0 ? 0 : R - s];
            const cplx<T> sb = self ? up : xt;      // mirror of element s
            b.x = __shfl_sync(0xffffffffu, sb.x, partner, L);
            b.y = __shfl_sync(0xffffffffu, sb.y, partner, L);
            x[s] = c2r_pre<T>(xs, b, twx[j + L * s]);
            x[R - 1 - s] = c2r_pre<T>(xt, a, twx[j + L * (R - 1 - s)]);
        } else {
            x[s] = c2r_pre_nomirror<T>(xs, twx[j + L * s]);
            x[R - 1 - s] = c2r_pre_dropped<T>(a, twx[j + L * (R - 1 - s)]);
        }
        carry = xs;
    }
}

}  // namespace
}  // namespace flusi
