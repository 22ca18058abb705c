// z passes in two register passes (colfft.cuh): the FP32 z transforms of zpass.cu
// at the lengths of FLUSI_COL_LENGTHS.  A tile is C consecutive columns q = jy Mxp + x:
// a full tile, or on grids whose full tiles would leave SMs idle 8 (up to 512 rows),
// with the same arithmetic.
//
// The inverse pass forms u and omega = i k x u from five transforms per column
// range (see k_zinv): W2 = Fz u_z; W4 = i (Fz(kz u_x) - kx W2); W0 = Fz u_x;
// W3 = i (ky W2 - Fz(kz u_y)); W1 = Fz u_y, W5 = i (kx W1 - ky W0).  They are five
// loads of one group, so the next component is on its way while this one is
// transformed and stored; the side rows W2 and W0 are read back by the threads
// that wrote them.
#include "colfft.cuh"

namespace flusi {
namespace {

template <int N> constexpr int z_cols() { return col_tile(N, 64); }
constexpr int kZSmall = 8;   // 64-byte rows, which L2 holds on grids that small

__device__ __forceinline__ unsigned long long evict_last()
{
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ unsigned long long evict_first()
{
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ unsigned long long evict_normal()
{
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// ---- forward: W[0..nf) in place, kept modes jz into rows jz of their columns
template <class X> struct ZForward {
    static constexpr int C = X::C, N = X::N, R = X::R;
    float2* W;
    const float2* tws;
    const CUtensorMap* map;
    int bh, Q, nqb, ntiles, Kz, Mz;
    size_t plane;

    __device__ __forceinline__ int tile_of(int i) const { return (int)(blockIdx.x + i * gridDim.x); }
    __device__ __forceinline__ bool exists(int i) const { return tile_of(i) < ntiles; }
    // rows h N/CH to (h + 1) N/CH of a tile
    __device__ __forceinline__ void issue(int i, int h, float2* buf, unsigned long long* bar) const
    {
        const int tile = tile_of(i), c = tile / nqb, q0 = (tile - c * nqb) * C;
        constexpr int half = N / X::CH;
        const int nb = half / bh;
        mbar_expect_tx(bar, (unsigned)(half * C * sizeof(float2)));
        for (int b = 0; b < nb; ++b) tma_load_3d(buf + b * bh * C, map, 2 * q0, h * half + b * bh, c, bar);
    }
    __device__ __forceinline__ void copy(int i, int h, float2* buf, int tid) const
    {
        const int tile = tile_of(i), c = tile / nqb;
        constexpr int lanes = C / 2, half = N / X::CH;
        const int col = (tid % lanes) * 2, q = (tile - c * nqb) * C + col;
        if (q >= Q) return;   // Q is a multiple of 4
        const float2* src = W + ((size_t)c * N + h * half) * plane + q;
        for (int z = tid / lanes; z < half; z += X::T / lanes) cp_async_16(buf + z * C + col, src + (size_t)z * plane);
    }
    struct Io {
        const ZForward& job;
        float2* base;
        int q0, f0;
        float2* out;
        bool ok;
        __device__ __forceinline__ void begin(int f, int col)
        {
            f0 = f;
            ok = q0 + col < job.Q;
            out = base + (ok ? q0 + col : 0);
        }
        __device__ __forceinline__ void all(const float2* a)
        {
            if (!ok) return;
#pragma unroll
            for (int i = 0; i < X::L; ++i) {   // modes |m| <= Kz only
                const int f = f0 + R * i, k = X::kept(R * i, R * i + R - 1);
                if (k == 0) continue;
                if (k == 2 || f <= job.Kz || f >= N - job.Kz)
                    out[(size_t)(2 * f <= N ? f : f - N + job.Mz) * job.plane] = a[i];
            }
        }
    };
    template <class Refill>
    __device__ __forceinline__ void work(int i, const typename X::Tile& t, int tid, int group, Refill refill) const
    {
        const int tile = tile_of(i), c = tile / nqb, q0 = (tile - c * nqb) * C;
        X::template first<false, false>(t, tws, tid, Kz, [](float2 v, int) { return v; });
        group_sync<X::T>(group);
        Io io{*this, W + (size_t)c * N * plane, q0, 0, nullptr, false};
        X::template second<false>(t, tid, io, refill);
    }
};

template <class X>
__global__ void __launch_bounds__(X::THREADS, X::MINB)
k_zcol_fwd(float2* __restrict__ W, Geom g, const double2* __restrict__ tw, int nf, const StepState* __restrict__ st,
           const __grid_constant__ CUtensorMap wmap, int bh, int* err, const Member* __restrict__ mb)
{
    if (mb) {   // one member of an ensemble batch (never with TMA)
        W = static_cast<float2*>(mb[blockIdx.z].W);
        st = mb[blockIdx.z].st;
        err = &mb[blockIdx.z].st->status;
    }
    const bool tma = bh > 0;
    if (block_leaves(st, tma ? err : nullptr)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ ColState state;
    float2* bufs = reinterpret_cast<float2*>(smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127));
    float2* tws = bufs + X::BUFS * X::BUF;
    const int Q = g.My * g.Mxp, nqb = ceil_div(Q, X::C);
    ZForward<X> job{W, tws, &wmap, bh, Q, nqb, nf * nqb, g.Kz, g.Mz, (size_t)g.ny * g.Mxp};
    X::table(tws, tw);
    col_loop<X>(bufs, state, tma, err, job);
}

// ---- inverse
template <class X> struct ZInverse {
    static constexpr int C = X::C, N = X::N, R = X::R, G = X::GROUPS, L = X::L;
    const float2* U;
    float2* W;
    const float2* tws;
    const CUtensorMap* map;
    int bh, Q, ntiles, phases, Kz, Mz, Mxp, Ky;
    size_t ustride, plane, field;          // strides of U's components, W's planes and fields
    float kxu, kyu, kzu;                   // 2 pi / L per axis

    // Load i is load k = i / G of its group: phase k % phases of the group's
    // (k / phases)-th column range.  Group 0 decides how many there are; a range
    // past the end is the last one again (the same values a second time).
    __device__ __forceinline__ bool exists(int i) const
    {
        return (int)(G * (blockIdx.x + (i / G / phases) * gridDim.x)) < ntiles;
    }
    __device__ __forceinline__ int q0_of(int i) const
    {
        const int tile = (int)(G * (blockIdx.x + (i / G / phases) * gridDim.x)) + i % G;
        return (tile < ntiles ? tile : ntiles - 1) * C;
    }
    __device__ __forceinline__ int phase_of(int i) const { return (i / G) % phases; }
    // u_z, u_x (weighted by kz), u_x, u_y (weighted), u_y; without vorticity u_x, u_y, u_z
    __device__ __forceinline__ int comp_of(int ph) const
    {
        return phases == 3 ? ph : ph == 0 ? 2 : ph <= 2 ? 0 : 1;
    }
    __device__ __forceinline__ void issue(int i, int h, float2* buf, unsigned long long* bar) const
    {
        constexpr int CH = X::CH, half = N / CH;
        const int q0 = q0_of(i), ph = phase_of(i), comp = comp_of(ph), kb = (Kz + 1) / bh;
        // the first of two reads of a component keeps its lines in L2
        const unsigned long long pol = phases == 3 ? evict_normal() : ph == 1 || ph == 3 ? evict_last() : evict_first();
        mbar_expect_tx(bar, (unsigned)((CH == 1 ? 2 : 1) * (Kz + 1) * C * sizeof(float2)));
        for (int b = 0; b < kb; ++b) {
            if (CH == 1 || h == 0) box(buf + b * bh * C, 2 * q0, b * bh, comp, bar, pol);
            if (CH == 1 || h == 1)
                box(buf + ((CH == 1 ? N : half) - Kz - 1 + b * bh) * C, 2 * q0, Kz + b * bh, comp, bar, pol);
        }
    }
    __device__ __forceinline__ void box(void* dst, int x, int row, int comp, unsigned long long* bar,
                                        unsigned long long pol) const
    {
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
            " [%0], [%1, {%2, %3, %4}], [%5], %6;\n" ::"r"(smem_u32(dst)),
            "l"(map), "r"(x), "r"(row), "r"(comp), "r"(smem_u32(bar)), "l"(pol)
            : "memory");
    }
    __device__ __forceinline__ void copy(int i, int h, float2* buf, int tid) const
    {
        constexpr int lanes = C / 2, half = N / X::CH;
        const int col = (tid % lanes) * 2, q = q0_of(i) + col;
        if (q >= Q) return;   // Q is a multiple of 4
        const float2* src = U + comp_of(phase_of(i)) * ustride + q;
        for (int o = tid / lanes; o < half; o += X::T / lanes) {
            const int s = h * half + o, jz = s <= Kz ? s : (s >= N - Kz ? s - N + Mz : -1);
            if (jz >= 0) cp_async_16(buf + o * C + col, src + (size_t)jz * Q);
        }
    }
    // A transform v of this phase: v itself to out_v (kept in L2 when it is a
    // later phase's side rows), and with a side field a the vorticity component
    // i (cv v + ca a) to out_c.
    struct Io {
        const ZInverse& job;
        int q0, ph;
        bool ok;
        size_t at;                           // this thread's column and first row
        float cv, ca;
        float2 *out_v, *out_c;
        const float2* side;
        unsigned long long pol;
        static constexpr int H = L > 18 ? (L + 3) / 4 : (L + 1) / 2;
        float2 a[H];                         // side rows of the next outputs

        __device__ __forceinline__ const float2* side_row(int i) const { return side + (at + (size_t)(R * i) * job.plane); }
        __device__ __forceinline__ float2 side_load(int i) const
        {
            float2 v;
            if (ph >= 3)   // the side rows' last use
                asm volatile("ld.global.cg.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(side_row(i)), "l"(pol));
            else v = __ldcg(side_row(i));
            return v;
        }
        __device__ __forceinline__ void begin(int f, int col)
        {
            const int q = q0 + col;
            ok = q < job.Q;
            const int qq = ok ? q : 0, jy = qq / job.Mxp, x = qq - jy * job.Mxp;
            at = (size_t)f * job.plane + qq;
            const float kx = job.kxu * float(x), ky = job.kyu * float(mode_of(jy, job.Ky));
            cv = ph == 1 ? 1.0f : ph == 3 ? -1.0f : kx;
            ca = ph == 1 ? -kx : ph == 3 ? ky : -ky;
            if (side && ok) {
#pragma unroll
                for (int i = 0; i < H; ++i) a[i] = side_load(i);
            }
        }
        __device__ __forceinline__ void all(const float2* v)
        {
            if (!ok) return;
            if (!side) {
#pragma unroll
                for (int i = 0; i < L; ++i)
                    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(out_v + (at + (size_t)(R * i) * job.plane)),
                                 "f"(v[i].x), "f"(v[i].y), "l"(pol)
                                 : "memory");
                return;
            }
#pragma unroll
            for (int i = 0; i < L; ++i) {
                if (i > 0 && i % H == 0) {
#pragma unroll
                    for (int u = 0; u < H && i + u < L; ++u) a[u] = side_load(i + u);
                }
                const size_t o = at + (size_t)(R * i) * job.plane;
                const float2 w = a[i % H];
                if (out_v) __stcs(out_v + o, v[i]);
                __stcs(out_c + o, cmuli(make_float2(cv * v[i].x + ca * w.x, cv * v[i].y + ca * w.y)));
            }
        }
    };
    template <class Refill>
    __device__ __forceinline__ void work(int i, const typename X::Tile& t, int tid, int group, Refill refill) const
    {
        const int ph = phase_of(i);
        const bool weighted = phases == 5 && (ph == 1 || ph == 3);
        X::template first<true, true>(t, tws, tid, Kz, [&](float2 v, int row) {
            return weighted ? cscale(v, kzu * float(2 * row <= N ? row : row - N)) : v;
        });
        group_sync<X::T>(group);
        Io io{*this, q0_of(i), ph};
        io.pol = phases == 3 ? evict_normal() : ph >= 3 ? evict_first() : evict_last();
        if (phases == 3) {
            io.out_v = W + ph * field;
            io.out_c = nullptr;
            io.side = nullptr;
        } else {
            io.out_v = ph == 0 ? W + 2 * field : ph == 2 ? W : ph == 4 ? W + field : nullptr;
            io.out_c = ph == 1 ? W + 4 * field : ph == 3 ? W + 3 * field : ph == 4 ? W + 5 * field : nullptr;
            io.side = ph == 1 || ph == 3 ? W + 2 * field : ph == 4 ? W : nullptr;
        }
        X::template second<true>(t, tid, io, refill);
    }
};

template <class X>
__global__ void __launch_bounds__(X::THREADS, X::MINB)
k_zcol_inv(const float2* __restrict__ U, float2* __restrict__ W, Geom g, const double2* __restrict__ tw, int nf,
           const StepState* __restrict__ st, const __grid_constant__ CUtensorMap umap, int bh, int* err,
           const Member* __restrict__ mb)
{
    if (mb) {   // one member of an ensemble batch (never with TMA)
        U = static_cast<const float2*>(mb[blockIdx.z].U);
        W = static_cast<float2*>(mb[blockIdx.z].W);
        st = mb[blockIdx.z].st;
        err = &mb[blockIdx.z].st->status;
    }
    const bool tma = bh > 0;
    if (block_leaves(st, tma ? err : nullptr)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ ColState state;
    float2* bufs = reinterpret_cast<float2*>(smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127));
    float2* tws = bufs + X::BUFS * X::BUF;
    const int Q = g.My * g.Mxp;
    const float two_pi = 6.283185307179586476925286766559f;
    const size_t plane = (size_t)g.ny * g.Mxp;
    ZInverse<X> job{U, W, tws, &umap, bh, Q, ceil_div(Q, X::C), nf < 6 ? 3 : 5, g.Kz, g.Mz, g.Mxp, g.Ky,
                    (size_t)g.Mz * Q, plane, (size_t)g.nz * plane,
                    two_pi / float(g.Lx), two_pi / float(g.Ly), two_pi / float(g.Lz)};
    X::table(tws, tw);
    col_loop<X>(bufs, state, tma, err, job);
}

}  // namespace

int zcol_full(int nz)
{
    switch (nz) {
#define FLUSI_CASE(n, R, L) case n: return z_cols<n>();
        FLUSI_COL_LENGTHS(FLUSI_CASE)
#undef FLUSI_CASE
    default: return 0;
    }
}

namespace {

template <class X>
cudaError_t launch_fwd(float2* W, int nf, const Geom& g, const double2* tw, const StepState* st, const CUtensorMap& map,
                       int bh, int* err, cudaStream_t s)
{
    const long long tiles = (long long)nf * ceil_div(g.My * g.Mxp, X::C);
    k_zcol_fwd<X><<<col_grid<X>(k_zcol_fwd<X>, tiles), X::THREADS, X::kSmem, s>>>(W, g, tw, nf, st, map, bh, err,
                                                                                 current_batch().mb);
    return cudaGetLastError();
}
template <class X>
cudaError_t launch_inv(const float2* U, float2* W, const Geom& g, const double2* tw, int nf, const StepState* st,
                       const CUtensorMap& map, int bh, int* err, cudaStream_t s)
{
    const long long tiles = ceil_div(ceil_div(g.My * g.Mxp, X::C), X::GROUPS);
    k_zcol_inv<X><<<col_grid<X>(k_zcol_inv<X>, tiles), X::THREADS, X::kSmem, s>>>(U, W, g, tw, nf, st, map, bh, err,
                                                                                 current_batch().mb);
    return cudaGetLastError();
}
// the small tile of a length that has one
template <int N> constexpr int z_small() { return N <= 512 ? kZSmall : z_cols<N>(); }

}  // namespace

cudaError_t launch_zcol_fwd(int cols, float2* W, int nf, const Geom& g, const double2* tw, const StepState* st,
                            const CUtensorMap& map, int bh, int* err, cudaStream_t s)
{
    switch (g.nz) {
#define FLUSI_CASE(n, R, L)                                                                                       \
    case n:                                                                                                       \
        return cols == z_cols<n>() ? launch_fwd<Col<R, L, z_cols<n>()>>(W, nf, g, tw, st, map, bh, err, s)         \
                                   : launch_fwd<Col<R, L, z_small<n>()>>(W, nf, g, tw, st, map, bh, err, s);
        FLUSI_COL_LENGTHS(FLUSI_CASE)
#undef FLUSI_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_zcol_inv(int cols, const float2* U, float2* W, const Geom& g, const double2* tw, int nf,
                            const StepState* st, const CUtensorMap& map, int bh, int* err, cudaStream_t s)
{
    switch (g.nz) {
#define FLUSI_CASE(n, R, L)                                                                                       \
    case n:                                                                                                       \
        return cols == z_cols<n>() ? launch_inv<Col<R, L, z_cols<n>()>>(U, W, g, tw, nf, st, map, bh, err, s)      \
                                   : launch_inv<Col<R, L, z_small<n>()>>(U, W, g, tw, nf, st, map, bh, err, s);
        FLUSI_COL_LENGTHS(FLUSI_CASE)
#undef FLUSI_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t configure_zcol(int nz)
{
    cudaError_t e = cudaSuccess;
    auto one = [&](const void* kernel, size_t smem) {
        if (!e) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
#define FLUSI_KERNELS(X)                                       \
    one((const void*)k_zcol_fwd<X>, X::kSmem);                 \
    one((const void*)k_zcol_inv<X>, X::kSmem);
    switch (nz) {
#define FLUSI_CASE(n, R, L)                                    \
    case n: {                                                  \
        using Full = Col<R, L, z_cols<n>()>;                   \
        using Small = Col<R, L, z_small<n>()>;                 \
        FLUSI_KERNELS(Full)                                    \
        FLUSI_KERNELS(Small)                                   \
        break;                                                 \
    }
        FLUSI_COL_LENGTHS(FLUSI_CASE)
#undef FLUSI_CASE
    }
#undef FLUSI_KERNELS
    return e;
}

}  // namespace flusi
