// x transforms of FP32 lines whose half length nh = nx/2 = R L is any product
// of 2s and 3s: register-resident like the square kernels of xpass.cu, with the
// two passes split unevenly over a warp.
//
// G lines at a time belong to one warp.  Pass 1 gives each line L lanes, lane j
// holding the R elements j + L t, t < R: the radix-R transform over t and the
// twiddles w_nh^{j q}.  Pass 2 gives each of the line's R rows q = n1 to one
// lane: the radix-L transform over j, which yields the point pairs n1 + R n2.
// The lanes of pass 2 are dealt over all G R rows of the warp's lines, so a
// length is served by an R and an L that fill both passes (384 = 2 x 24 x 8:
// four lines of 8 lanes, then 96 rows over 32 lanes in three rounds) rather
// than by one R for both.  Between the passes the values go through the line's
// slice in shared memory (element j of row q at q LP + j, LP odd), which only
// the warp touches: __syncwarp is enough.  Pass 2 works in place, so a row's
// values keep their slots and the rounds do not wait for each other.
//
// The forward transform runs the same steps transposed, in reverse.  The c2r
// and r2c steps pair element t of lane j with element R-1-t of lane L-j (lane
// 0: its own element R-t), by shuffles; elements that the 2/3 rule drops on
// every lane (t >= NT) are neither loaded, exchanged nor stored.
//
// What bounds it: shared-memory wavefronts and instruction issue, as for the
// square kernels; the general shared-memory kernel (k_xpass) that served these
// lengths goes through shared memory once per radix-8/4/3 stage.  Measured,
// FP32, k_xpass -> these: physical pass 384 x 384 x 768 3.27 -> 1.25 ms (3.1 GB
// of lines: 2.5 TB/s), 192^3 233 -> 90 us, 162 x 81 x 243 133 -> 49 us,
// 48 x 36 x 24 33 -> 18 us; sponge lines 384 x 384 x 768 2.07 -> 0.52 ms;
// set_state and get_state at 512^3 3.36 and 2.23 -> 1.33 and 0.94 ms, at
// 1024^3 29.1 and 19.8 -> 10.6 and 8.1 ms (their z and y passes included, which
// became faster too).
#pragma once

#include "fft.cuh"
#include "kernels.cuh"
#include "xphys.cuh"

namespace flusi {
namespace {

template <int R_, int L_, int G_> struct XLine {
    static constexpr int R = R_, L = L_, G = G_, NH = R * L;
    static constexpr int LP = L | 1;                       // row pitch in a slice
    static constexpr int ROUNDS = (G * R + 31) / 32;       // pass 2
    // lanes of pass 1 and rows of pass 2 that meet a bank pair of an earlier one, both
    // over half-warps of 16, for slices cs apart
    static constexpr int conflicts(int cs)
    {
        int n = 0;
        for (int pass = 0; pass < 2; ++pass) {
            const int per = pass ? R : L, step = pass ? LP : 1, all = G * per;
            for (int h = 0; h < all; h += 16) {
                unsigned seen = 0;
                for (int i = h; i < all && i < h + 16; ++i) {
                    const unsigned bit = 1u << (((i / per) * cs + (i % per) * step) & 15);
                    n += (seen & bit) ? 1 : 0;
                    seen |= bit;
                }
            }
        }
        return n;
    }
    static constexpr int slice()
    {
        int best = R * LP, low = conflicts(best);
        for (int cs = R * LP + 1; cs < R * LP + 16; ++cs)
            if (conflicts(cs) < low) {
                low = conflicts(cs);
                best = cs;
            }
        return best;
    }
    static constexpr int CS = slice();
    // elements per lane that can be a stored mode (k < Mxp, Mx padded to 4)
    static constexpr int MXP = (2 * NH / 3 + 1 + 3) / 4 * 4;
    static constexpr int NT = (MXP - 1) / L + 1 < R ? (MXP - 1) / L + 1 : R;
    static constexpr int NA = sq_always<R, L>();           // elements that are kept modes on every lane

    static_assert(G * L <= 32, "a warp's lines");

    // where this lane stands in pass 1
    struct Lane {
        int g, j, partner;
        bool on;
    };
    __device__ __forceinline__ static Lane lane_of(int lane)
    {
        Lane p;
        p.g = lane / L;
        p.j = lane - p.g * L;
        p.on = G * L == 32 || p.g < G;
        if (!p.on) p.g = 0;
        p.partner = p.on ? p.g * L + (p.j == 0 ? 0 : L - p.j) : lane;
        return p;
    }

    __device__ __forceinline__ static float2 from(float2 v, int src)
    {
        return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
    }

    // x[t] = X[j + L t] -> Z[j + L t].  From the middle outwards, so that every
    // element read is still the original one (element s + 1, overwritten the
    // step before, is carried).
    __device__ __forceinline__ static void pre(float2* x, const Lane& p, const float2* twx)
    {
        const bool self = p.j == 0;
        const float2 zero = make_float2(0.0f, 0.0f);
        float2 carry = x[R / 2];
        if constexpr (R % 2 == 1) {
            constexpr int m = R / 2;      // its own mirror on the partner lane
            if constexpr (m < NT || m + 1 < NT) {
                const float2 o = from(self ? (m + 1 < R ? x[m + 1 < R ? m + 1 : m] : zero) : x[m], p.partner);
                x[m] = c2r_pre<float>(x[m], o, twx[p.j + L * m]);
            }
        }
#pragma unroll
        for (int s = R / 2 - 1; s >= 0; --s) {
            const int q = R - 1 - s;
            const float2 xs = x[s], xq = x[q];
            const float2 a = from(self ? carry : xs, p.partner);     // mirror of element q
            if (q < NT) {
                const float2 up = s == 0 ? zero : x[s == 0 ? 0 : R - s];
                const float2 b = from(self ? up : xq, p.partner);    // mirror of element s
                x[s] = c2r_pre<float>(xs, b, twx[p.j + L * s]);
                x[q] = c2r_pre<float>(xq, a, twx[p.j + L * q]);
            } else {
                x[s] = c2r_pre_nomirror<float>(xs, twx[p.j + L * s]);
                x[q] = c2r_pre_dropped<float>(a, twx[p.j + L * q]);
            }
            carry = xs;
        }
    }

    // Modes -> rows in the slices.  src: this lane's line of Mx kept modes (any
    // line of the grid where the values are not used).
    __device__ __forceinline__ static void inverse_pass1(float2* slices, const Lane& p, const float2* twx,
                                                         const float2* tw2, const float2* src, int Mx)
    {
        float2 v[R];
#pragma unroll
        for (int t = 0; t < R; ++t)
            v[t] = t < NA ? src[p.j + L * t] : t < NT && p.j + L * t < Mx ? src[p.j + L * t] : make_float2(0.0f, 0.0f);
        if (p.j == 0) v[0].y = 0.0f;       // a real line has a real mean
        pre(v, p, twx);
        Dft<float, R, true>::run(v);
#pragma unroll
        for (int q = 1; q < R; ++q) v[q] = cmul(v[q], cconj(tw2[q * LP + p.j]));
        if (p.on) {
            float2* s = slices + p.g * CS + p.j;
#pragma unroll
            for (int q = 0; q < R; ++q) s[q * LP] = v[q];
        }
    }

    // Calls each(slot of row n1, line g, n1) for this lane's rows of pass 2.
    template <class Each> __device__ __forceinline__ static void rows(float2* slices, int lane, Each each)
    {
#pragma unroll 1
        for (int u = lane; u < G * R; u += 32) {
            const int g = u / R, n1 = u - g * R;
            each(slices + g * CS + n1 * LP, g, n1);
        }
    }
    __device__ __forceinline__ static void get(const float2* s, float2* a)
    {
#pragma unroll
        for (int i = 0; i < L; ++i) a[i] = s[i];
    }
    __device__ __forceinline__ static void put(float2* s, const float2* a)
    {
#pragma unroll
        for (int i = 0; i < L; ++i) s[i] = a[i];
    }
    // forward pass 2 of row n1: the pairs n1 + R i in a[i], left in the slot
    __device__ __forceinline__ static void forward_row(float2* s, int n1, float2* a, const float2* tw2)
    {
        Dft<float, L, false>::run(a);
#pragma unroll
        for (int i = 1; i < L; ++i) a[i] = cmul(a[i], tw2[n1 * LP + i]);
        put(s, a);
    }

    // Rows in the slices -> modes of this lane's line `out` (stored where ok).
    __device__ __forceinline__ static void forward_pass1(const float2* slices, const Lane& p, const float2* twx, float2* out,
                                                         bool ok, int Mx, int Mxp)
    {
        float2 v[R];
        const float2* s = slices + p.g * CS + p.j;
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = s[q * LP];
        Dft<float, R, false>::run(v);      // v[q] = Z[j + L q]
#pragma unroll
        for (int q = 0; q < NT; ++q) {
            const float2 o = from(v[R - 1 - q], p.partner);
            const float2 m = p.j != 0 ? o : v[(R - q) % R];
            const int k = p.j + L * q;
            const float2 x = q < NA || k < Mx ? r2c_post<float>(v[q], m, twx[k]) : make_float2(0.0f, 0.0f);
            if (ok && (q < NA || k < Mxp)) out[k] = x;
        }
    }

    // shared tables: w_nx^k, k < nh, then w_nh^{q j} at q LP + j
    static constexpr int TABLE = NH + R * LP;
    __device__ __forceinline__ static void tables(float2* twx, const double2* tw, int nx)
    {
        const float2* w = reinterpret_cast<const float2*>(tw + nx);   // the FP32 copy
        float2* tw2 = twx + NH;
        for (int i = threadIdx.x; i < NH; i += blockDim.x) {
            twx[i] = w[i];
            const int q = i / L, j = i - q * L;
            tw2[q * LP + j] = w[(2 * q * j) % nx];
        }
    }
};

// ---- set_state, get_state and the separate sponge pass: lines on their own,
// G per warp, no block barrier after the tables.
template <class X, int MODE>
__global__ void __launch_bounds__(128)
k_xlines(float2* __restrict__ W, Geom g, const double2* __restrict__ tw, XExtra ex, int wide)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* twx = reinterpret_cast<float2*>(smem_raw);
    float2* tw2 = twx + X::NH;
    X::tables(twx, tw, g.nx);
    __syncthreads();
    constexpr int R = X::R, L = X::L, G = X::G;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = blockDim.x / 32;
    float2* slices = twx + X::TABLE + warp * G * X::CS;
    const auto p = X::lane_of(lane);
    const int nrows = g.nz * g.ny, Mx = g.Mx, Mxp = g.Mxp;
    const long long lines = (long long)ex.ncomp * nrows;
#pragma unroll 1
    for (long long l0 = ((long long)blockIdx.x * nw + warp) * G; l0 < lines; l0 += (long long)gridDim.x * nw * G) {
        const long long ln = l0 + p.g;
        const bool ok = p.on && ln < lines;
        float2* modes = W + ((size_t)ex.comp0 * nrows + (size_t)(ok ? ln : l0)) * Mxp;
        if (MODE != XP_R2C) {
            X::inverse_pass1(slices, p, twx, tw2, modes, Mx);
            __syncwarp();
        }
        X::rows(slices, lane, [&](float2* s, int gl, int n1) {
            const long long line = l0 + gl;
            float2 a[L];
            if (MODE != XP_R2C) {
                X::get(s, a);
                Dft<float, L, true>::run(a);
            }
            if (MODE == XP_SPONGE) {   // chi_sp omega (Sec. 2.3): keep the points of the sponge slabs
                const int r = (int)(line % nrows), z = r / g.ny, y = r - z * g.ny;
                const bool in_row = y >= ex.sponge0[1] || z >= ex.sponge0[2];
#pragma unroll
                for (int i = 0; i < L; ++i) {
                    const int x = 2 * (n1 + R * i);
                    if (!in_row && x < ex.sponge0[0]) a[i].x = 0.0f;
                    if (!in_row && x + 1 < ex.sponge0[0]) a[i].y = 0.0f;
                }
                X::forward_row(s, n1, a, tw2);
                return;
            }
            // the real line of this slice: point pairs n1 + R i
            const long long f = line / nrows, o = f * ex.cstride + (line - f * nrows) * (long long)(2 * X::NH) + 2 * n1;
            const bool on = line < lines;
            if (MODE == XP_R2C) {
#pragma unroll
                for (int i = 0; i < L; ++i) {
                    a[i] = make_float2(0.0f, 0.0f);
                    if (!on) continue;
                    if (ex.real_fp64) {
                        const double* d = static_cast<const double*>(ex.rin) + o + 2 * R * i;
                        a[i] = make_float2(float(d[0]), float(d[1]));
                    } else {
                        const float* d = static_cast<const float*>(ex.rin) + o + 2 * R * i;
                        a[i] = wide ? *reinterpret_cast<const float2*>(d) : make_float2(d[0], d[1]);
                    }
                }
                X::forward_row(s, n1, a, tw2);
            } else if (on) {
#pragma unroll
                for (int i = 0; i < L; ++i) {
                    if (ex.real_fp64) {
                        double* d = static_cast<double*>(ex.rout) + o + 2 * R * i;
                        d[0] = double(a[i].x);
                        d[1] = double(a[i].y);
                    } else {
                        float* d = static_cast<float*>(ex.rout) + o + 2 * R * i;
                        if (wide) {
                            *reinterpret_cast<float2*>(d) = a[i];
                        } else {
                            d[0] = a[i].x;
                            d[1] = a[i].y;
                        }
                    }
                }
            }
        });
        __syncwarp();
        if (MODE != XP_C2R) {
            X::forward_pass1(slices, p, twx, modes, ok, Mx, Mxp);
            __syncwarp();
        }
    }
}

// ---- the physical x pass: as k_xpass_sq (xpass.cu), with this file's lines.
// Three warps; a tile is RB = G rows, of which every warp inverse-transforms
// 2 G of the 6 G lines and forward-transforms G of the 3 G.
template <class X, int MINB>
__global__ void __launch_bounds__(96, MINB)
k_xline_phys(float2* __restrict__ W, Geom g, const double2* __restrict__ tw, XExtra ex,
             const StepState* __restrict__ st, const Member* __restrict__ mb)
{
    if (mb) {   // one member of an ensemble batch
        const Member& m = mb[blockIdx.z];
        W = static_cast<float2*>(m.W);
        st = m.st;
        ex.frame = m.fr;
        ex.part = m.part;
    }
    const bool failed = step_failed(st);
    constexpr int NT = 96, NW = 3;
    constexpr int R = X::R, L = X::L, G = X::G, NH = X::NH, CS = X::CS, LP = X::LP;
    constexpr int RB = G, NG = NW * G;         // rows of a tile, lane groups of the block
    // lengths whose sponge runs in a square kernel (xpass.cu): those refuse a state
    // whose energy overflows, and so does this one
    constexpr bool ENERGY = NH == 32 || NH == 64 || NH == 128;
    const int Mx = g.Mx, Mxp = g.Mxp;
    const int nrows = g.nz * g.ny;
    const int ntiles = ceil_div(nrows, RB);

    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* wacc = reinterpret_cast<double*>(smem_raw);                    // [warps][36]
    FrameT<float>* Fs = reinterpret_cast<FrameT<float>*>(wacc + NW * 36);
    float2* twx = reinterpret_cast<float2*>(reinterpret_cast<unsigned char*>(Fs) + align16(sizeof(FrameT<float>)));
    float2* tw2 = twx + NH;
    float2* buf = twx + X::TABLE;              // 6 RB line slices, line (field f, row rr) at f RB + rr
    __shared__ int rowmask[RB];

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    X::tables(twx, tw, g.nx);
    load_frame_t<float>(Fs, ex.frame);
    if (__syncthreads_or(failed)) return;
    const auto p = X::lane_of(lane);
    const float dxT = float(g.dx), dyT = float(g.dy), dzT = float(g.dz);
    const FrameT<float>& F = *Fs;
    const bool layer = ex.layer0[0] < g.nx || ex.layer0[1] < g.ny || ex.layer0[2] < g.nz;
    const float uinf[3] = {float(ex.u_inf[0]), float(ex.u_inf[1]), float(ex.u_inf[2])};

    const int P = ex.nvirt;   // virtual CTAs: see k_xpass_sq
#pragma unroll 1
    for (int vb = blockIdx.x; vb < P; vb += gridDim.x) {
        for (int i = tid; i < NW * 36; i += NT) wacc[i] = 0.0;
        __syncthreads();
        double e_acc = 0.0;
        float m_acc = 0.0f;
        int bad = 0;
#pragma unroll 1
        for (int tile = vb; tile < ntiles; tile += P) {
            const int row0 = tile * RB;
            if (tid < 6) {   // the next tile's input lines on their way into L2
                const long long next0 = (long long)(tile + P) * RB;
                if (next0 < nrows) {
                    const int nr = min(RB, nrows - (int)next0);
                    prefetch_l2_bulk(W + ((size_t)tid * nrows + next0) * Mxp, (unsigned)(nr * Mxp * sizeof(float2)));
                }
            }
            if (tid < RB) {
                const int r = row0 + tid;
                int mask = 0;
                if (r < nrows) {
                    const int z = r / g.ny, y = r - z * g.ny;
                    const float Y = float(y) * dyT, Z = float(z) * dzT;
                    for (int q = 0; q < 3; ++q)
                        if (F.active[q] && Y >= F.box[q][2] && Y <= F.box[q][3] && Z >= F.box[q][4] && Z <= F.box[q][5])
                            mask |= 1 << q;
                }
                rowmask[tid] = mask;
            }
#pragma unroll 1
            for (int li = 0; li < 2; ++li) {
                const int c0 = warp * G + li * NG, cl = c0 + p.g;
                const int r = row0 + cl % RB;
                const bool ok = p.on && r < nrows;
                const float2* src = W + ((size_t)(cl / RB) * nrows + (ok ? r : 0)) * Mxp;
                float2* slices = buf + c0 * CS;
                X::inverse_pass1(slices, p, twx, tw2, src, Mx);
                __syncwarp();
                X::rows(slices, lane, [&](float2* s, int, int) {
                    float2 a[L];
                    X::get(s, a);
                    Dft<float, L, true>::run(a);
                    X::put(s, a);
                });
            }
            __syncthreads();

            // physical space: NL = u x omega into the omega lines, energy and
            // max |u|^2, a point pair per thread.  An NL value that is not finite
            // turns `odd` into NaN (0 times it).  A u that is not makes the energy
            // sum so, but a large finite u does too: then the values are looked at.
            float2 e2 = make_float2(0.0f, 0.0f), odd = make_float2(0.0f, 0.0f);
#pragma unroll 2
            for (int i = tid; i < RB * NH; i += NT) {
                const int rr = i / NH, lrow = i - rr * NH;
                if (row0 + rr >= nrows) continue;
                const int n1 = lrow / L, n2 = lrow - n1 * L, slot = n1 * LP + n2;
                float2 u[3], w[3], nl[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    u[q] = buf[(q * RB + rr) * CS + slot];
                    w[q] = buf[((3 + q) * RB + rr) * CS + slot];
                }
                cross3_pair(u, w, nl);
                if (layer) {   // Dirichlet layer u = u_inf (Sec. 2.3)
                    const int r = row0 + rr, z = r / g.ny, y = r - z * g.ny, x = 2 * (n1 + R * n2);
                    const bool in_row = y >= ex.layer0[1] || z >= ex.layer0[2];
                    if (in_row || x >= ex.layer0[0]) {
#pragma unroll
                        for (int q = 0; q < 3; ++q) nl[q].x -= F.inv_eta * (u[q].x - uinf[q]);
                    }
                    if (in_row || x + 1 >= ex.layer0[0]) {
#pragma unroll
                        for (int q = 0; q < 3; ++q) nl[q].y -= F.inv_eta * (u[q].y - uinf[q]);
                    }
                }
                const float2 uu = __ffma2_rn(u[2], u[2], __ffma2_rn(u[1], u[1], __fmul2_rn(u[0], u[0])));
                e2 = __fadd2_rn(e2, uu);
                m_acc = fmaxf(m_acc, fmaxf(uu.x, uu.y));
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    buf[((3 + q) * RB + rr) * CS + slot] = nl[q];
                    odd = __ffma2_rn(nl[q], make_float2(0.0f, 0.0f), odd);
                }
            }
            const float e_tile = e2.x + e2.y;
            e_acc += double(e_tile);
            float odd_tile = odd.x + odd.y;
            if (!isfinite(e_tile)) {
                if (ENERGY) bad = 1;
                for (int i = tid; i < RB * NH; i += NT) {
                    const int rr = i / NH, lrow = i - rr * NH;
                    if (row0 + rr >= nrows) continue;
                    for (int q = 0; q < 3; ++q) {
                        const float2 u = buf[(q * RB + rr) * CS + lrow / L * LP + lrow % L];
                        if (!isfinite(u.x) || !isfinite(u.y)) bad = 1;
                    }
                }
            }

            // penalization, only in tiles with a row that meets a part's box
            int tile_any = 0;
#pragma unroll
            for (int rr = 0; rr < RB; ++rr) tile_any |= rowmask[rr];
            if (tile_any) {   // uniform over the block
                __syncthreads();
                constexpr int NX = 2 * NH;
#pragma unroll 1
                for (int i0 = 0; i0 < RB * NX; i0 += NT) {
                    const int i = i0 + tid;
                    const int rr = i / NX, xi = i - rr * NX;
                    const int r = row0 + rr;
                    const int mask = (i < RB * NX && r < nrows) ? rowmask[rr] : 0;
                    float chi = 0.0f, us[3] = {0.0f, 0.0f, 0.0f}, Xp[3] = {0.0f, 0.0f, 0.0f}, u[3] = {0.0f, 0.0f, 0.0f};
                    int colr = 0;
                    if (mask != 0) {
                        const int z = r / g.ny, y = r - z * g.ny;
                        Xp[0] = float(xi) * dxT;
                        Xp[1] = float(y) * dyT;
                        Xp[2] = float(z) * dzT;
                        const bool inrow[3] = {(mask & 1) != 0, (mask & 2) != 0, (mask & 4) != 0};
                        solid_at(F, Xp, inrow, chi, colr, us);
                        if (chi > 0.0f) {
                            // point xi is half h of the pair n1 + R n2
                            const int pp = xi >> 1, h = xi & 1, n2 = pp / R, slot = (pp - n2 * R) * LP + n2;
                            const float pen = chi * F.inv_eta;
#pragma unroll
                            for (int q = 0; q < 3; ++q) {
                                const float* ul = reinterpret_cast<const float*>(buf + (q * RB + rr) * CS + slot);
                                float* nl = reinterpret_cast<float*>(buf + ((3 + q) * RB + rr) * CS + slot);
                                u[q] = ul[h];
                                nl[h] -= pen * (u[q] - us[q]);
                                odd_tile = __fmaf_rn(nl[h], 0.0f, odd_tile);
                            }
                        }
                    }
                    if (__any_sync(0xffffffffu, colr != 0)) {
                        for (int cc = 0; cc < 3; ++cc) {
                            const bool has = colr == cc + 1;
                            if (!__any_sync(0xffffffffu, has)) continue;
                            float acc[12];   // this lane's point in FP32, the sums above in FP64 or closer
#pragma unroll
                            for (int k2 = 0; k2 < 12; ++k2) acc[k2] = 0.0f;
                            if (has) {
                                const float* ref = cc == 0 ? F.xc : F.pv[cc - 1];
                                const float rv[3] = {Xp[0] - ref[0], Xp[1] - ref[1], Xp[2] - ref[2]};
                                float pu[3], cu[3];
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    pu[q] = chi * (u[q] - us[q]);
                                    cu[q] = chi * us[q];
                                    acc[q] = pu[q];
                                    acc[6 + q] = cu[q];
                                }
                                cross3(rv, pu, acc + 3);
                                cross3(rv, cu, acc + 9);
                            }
                            warp_sums12(acc, wacc + warp * 36 + cc * 12, lane);
                        }
                    }
                }
            }
            if (!(odd_tile == 0.0f)) bad = 1;
            __syncthreads();

            // forward on the three NL lines of each row, one per lane group
            {
                const int c0 = warp * G, cl = c0 + p.g;
                const int r = row0 + cl % RB;
                const bool ok = p.on && r < nrows;
                float2* slices = buf + (3 * RB + c0) * CS;
                X::rows(slices, lane, [&](float2* s, int, int n1) {
                    float2 a[L];
                    X::get(s, a);
                    X::forward_row(s, n1, a, tw2);
                });
                __syncwarp();
                float2* out = W + ((size_t)(cl / RB) * nrows + (ok ? r : 0)) * Mxp;
                X::forward_pass1(slices, p, twx, out, ok, Mx, Mxp);
            }
            // no block barrier before the next tile: a warp's next inverse
            // lines are u lines (their readers are behind the barrier above)
            // and its own forward lines (3 RB = NG)
            __syncwarp();
        }

        __shared__ double red[NW][3];
        e_acc = warp_sum(e_acc);
        double m_d = double(m_acc);
        for (int o = 16; o > 0; o >>= 1) m_d = fmax(m_d, __shfl_xor_sync(0xffffffffu, m_d, o));
        const int anybad = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            red[warp][0] = e_acc;
            red[warp][1] = m_d;
            red[warp][2] = anybad ? 1.0 : 0.0;
        }
        __syncthreads();
        double* outp = ex.part + (size_t)vb * kNumSums;
        if (tid < 36) {
            double s2 = 0.0;
            for (int w = 0; w < NW; ++w) s2 += wacc[w * 36 + tid];
            outp[tid] = s2;
        } else if (tid == kSumEkin) {
            double s2 = 0.0;
            for (int w = 0; w < NW; ++w) s2 += red[w][0];
            outp[tid] = s2;
        } else if (tid == kSumUmax2 || tid == kSumBad) {
            double s2 = 0.0;
            for (int w = 0; w < NW; ++w) s2 = fmax(s2, red[w][tid == kSumUmax2 ? 1 : 2]);
            outp[tid] = s2;
        } else if (tid < kNumSums) {
            outp[tid] = 0.0;
        }
        __syncthreads();   // wacc and red read before the next virtual CTA clears them
    }
}

// blocks per SM that the registers are capped for: R complex values a lane and
// what the transform of R needs beside them
template <int R> constexpr int xline_minb() { return R <= 12 ? 8 : R <= 18 ? 6 : 5; }

template <class X> constexpr size_t xline_phys_smem()
{
    return sizeof(double) * 3 * 36 + align16(sizeof(FrameT<float>)) +
           sizeof(float2) * ((size_t)X::TABLE + (size_t)6 * X::G * X::CS);
}
template <class X> constexpr size_t xline_lines_smem(int warps)
{
    return sizeof(float2) * ((size_t)X::TABLE + (size_t)warps * X::G * X::CS);
}

}  // namespace

// What a length's kernels offer (one entry per nx, made in the xline_*.cu files).
struct XLineOps {
    int nx, rows;                                         // rows of a physical tile
    int (*phys_per_sm)();                                 // resident physical CTAs per SM
    void (*phys)(dim3 grid, cudaStream_t s, float2* W, const Geom& g, const double2* tw, const XExtra& ex,
                 const StepState* st, const Member* mb);
    void (*lines)(int mode, cudaStream_t s, float2* W, const Geom& g, const double2* tw, const XExtra& ex, int sms);
    cudaError_t (*configure)();
};

namespace {

template <class X> struct XLineOf {
    static constexpr int MINB = xline_minb<X::R>();
    static int phys_per_sm()
    {
        int n = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_xline_phys<X, MINB>, 96, xline_phys_smem<X>());
        return n;
    }
    static void phys(dim3 grid, cudaStream_t s, float2* W, const Geom& g, const double2* tw, const XExtra& ex,
                     const StepState* st, const Member* mb)
    {
        k_xline_phys<X, MINB><<<grid, 96, xline_phys_smem<X>(), s>>>(W, g, tw, ex, st, mb);
    }
    template <int MODE>
    static void one(cudaStream_t s, float2* W, const Geom& g, const double2* tw, const XExtra& ex, int sms)
    {
        constexpr int warps = 4;
        constexpr size_t smem = xline_lines_smem<X>(warps);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_xlines<X, MODE>, 32 * warps, smem);
        const long long lines = (long long)ex.ncomp * g.ny * g.nz;
        const long long want = (lines + warps * X::G - 1) / (warps * X::G), most = (long long)sms * (per_sm > 0 ? per_sm : 1);
        // pairs of real values move at once where every pair is aligned (a row
        // holds an even number of them)
        const uintptr_t real = reinterpret_cast<uintptr_t>(MODE == XP_C2R ? ex.rout : ex.rin);
        const int wide = real % 8 == 0 && ex.cstride % 2 == 0;
        k_xlines<X, MODE><<<(int)(want < most ? want : most), 32 * warps, smem, s>>>(W, g, tw, ex, wide);
    }
    static void lines(int mode, cudaStream_t s, float2* W, const Geom& g, const double2* tw, const XExtra& ex, int sms)
    {
        if (mode == XP_R2C) one<XP_R2C>(s, W, g, tw, ex, sms);
        else if (mode == XP_C2R) one<XP_C2R>(s, W, g, tw, ex, sms);
        else one<XP_SPONGE>(s, W, g, tw, ex, sms);
    }
    static cudaError_t configure_lines()
    {
        constexpr int b = (int)xline_lines_smem<X>(4);
        cudaError_t e = cudaSuccess;
        if (!e) e = cudaFuncSetAttribute(k_xlines<X, XP_R2C>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
        if (!e) e = cudaFuncSetAttribute(k_xlines<X, XP_C2R>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
        if (!e) e = cudaFuncSetAttribute(k_xlines<X, XP_SPONGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, b);
        return e;
    }
    static cudaError_t configure()
    {
        const cudaError_t e = cudaFuncSetAttribute(k_xline_phys<X, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)xline_phys_smem<X>());
        return e ? e : configure_lines();
    }
    static constexpr XLineOps all() { return {2 * X::NH, X::G, phys_per_sm, phys, lines, configure}; }
    // lengths whose physical pass has a square or rectangular kernel of its own (xpass.cu)
    static constexpr XLineOps lines_only() { return {2 * X::NH, 0, nullptr, nullptr, lines, configure_lines}; }
};

}  // namespace
}  // namespace flusi
