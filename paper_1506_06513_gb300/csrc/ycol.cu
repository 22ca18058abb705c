// y passes in two register passes (colfft.cuh): the FP32 y transforms of
// ypass.cu at the lengths of FLUSI_COL_LENGTHS.  A tile is 16
// consecutive x modes of NP consecutive z planes of one component.
#include "colfft.cuh"

namespace flusi {
namespace {

template <int N> constexpr int y_cols() { return col_tile(N, 256); }
constexpr int kTX = 16;   // x modes of a tile, 128-byte rows

template <class X, bool INV> struct YJob {
    static constexpr int C = X::C, N = X::N, R = X::R, TX = kTX, NP = C / TX;
    float2* W;
    const float2* tws;
    const CUtensorMap* map;
    int bh, nz, Mxp, Ky, My, nxb, nzb, ntiles;
    size_t plane;

    __device__ __forceinline__ int tile_of(int i) const { return (int)(blockIdx.x + i * gridDim.x); }
    __device__ __forceinline__ bool exists(int i) const { return tile_of(i) < ntiles; }
    __device__ __forceinline__ void where(int i, int& x0, int& z0, int& c) const
    {
        const int tile = tile_of(i), b = tile / nxb;
        x0 = (tile - b * nxb) * TX;
        c = b / nzb;
        z0 = (b - c * nzb) * NP;
    }
    // boxes of bh rows of NP planes of TX columns: rows h N/CH to (h+1) N/CH.
    // Inverse: modes 0..Ky to rows 0..Ky, modes Ky..2Ky to rows N-Ky-1..N-1 (row
    // N-Ky-1, a dropped mode, is not read).
    __device__ __forceinline__ void issue(int i, int h, float2* buf, unsigned long long* bar) const
    {
        constexpr int CH = X::CH, half = N / CH;
        int x0, z0, c;
        where(i, x0, z0, c);
        const int pl = c * nz + z0;
        const unsigned box = (unsigned)(bh * C * sizeof(float2));
        if (INV) {
            const int kb = (Ky + 1) / bh;
            mbar_expect_tx(bar, (CH == 1 ? 2 : 1) * kb * box);
            for (int q = 0; q < kb; ++q) {
                if (CH == 1 || h == 0) tma_load_3d(buf + q * bh * C, map, 2 * x0, pl, q * bh, bar);
                if (CH == 1 || h == 1)
                    tma_load_3d(buf + ((CH == 1 ? N : half) - Ky - 1 + q * bh) * C, map, 2 * x0, pl, Ky + q * bh, bar);
            }
        } else {
            const int nb = half / bh;
            mbar_expect_tx(bar, nb * box);
            for (int q = 0; q < nb; ++q) tma_load_3d(buf + q * bh * C, map, 2 * x0, pl, h * half + q * bh, bar);
        }
    }
    // the same rows by 16-byte copies, two columns each (columns outside the
    // grid are left as they are: nothing of them is stored)
    __device__ __forceinline__ void copy(int i, int h, float2* buf, int tid) const
    {
        int x0, z0, c;
        where(i, x0, z0, c);
        constexpr int lanes = C / 2, half = N / X::CH;
        const int col = (tid % lanes) * 2, z = z0 + col / TX, x = x0 + col % TX;
        if (z >= nz || x >= Mxp) return;   // Mxp is a multiple of 4
        const float2* src = W + ((size_t)c * nz + z) * plane + x;
        for (int o = tid / lanes; o < half; o += X::T / lanes) {
            const int s = h * half + o, j = INV ? (s <= Ky ? s : (s >= N - Ky ? s - N + My : -1)) : s;
            if (j >= 0) cp_async_16(buf + o * C + col, src + (size_t)j * Mxp);
        }
    }
    struct Io {
        const YJob& job;
        float2* base;
        int x0, z0, q;
        float2* out;
        bool ok;
        __device__ __forceinline__ void begin(int q_, int col)
        {
            const int z = z0 + col / TX, x = x0 + col % TX;
            q = q_;
            ok = z < job.nz && x < job.Mxp;
            out = base + (size_t)(ok ? z : 0) * job.plane + (ok ? x : 0);
        }
        __device__ __forceinline__ void all(const float2* a)
        {
            if (!ok) return;
#pragma unroll
            for (int i = 0; i < X::L; ++i) {
                const int f = q + R * i;
                if (INV) {
                    out[(size_t)f * job.Mxp] = a[i];
                } else {   // modes |m| <= Ky only
                    const int k = X::kept(R * i, R * i + R - 1);
                    if (k == 0) continue;
                    if (k == 2 || f <= job.Ky || f >= N - job.Ky)
                        out[(size_t)(2 * f <= N ? f : f - N + job.My) * job.Mxp] = a[i];
                }
            }
        }
    };
    template <class Refill>
    __device__ __forceinline__ void work(int i, const typename X::Tile& t, int tid, int group, Refill refill) const
    {
        int x0, z0, c;
        where(i, x0, z0, c);
        X::template first<INV, INV>(t, tws, tid, Ky, [](float2 v, int) { return v; });
        group_sync<X::T>(group);
        Io io{*this, W + (size_t)c * nz * plane, x0, z0, 0, nullptr, false};
        X::template second<INV>(t, tid, io, refill);
    }
};

template <class X, bool INV>
__global__ void __launch_bounds__(X::THREADS, X::MINB)
k_ycol(float2* __restrict__ W, Geom g, const double2* __restrict__ tw, int ncomp, const StepState* __restrict__ st,
       const __grid_constant__ CUtensorMap tmap, int bh, int* err, const Member* __restrict__ mb)
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
    // the tiles at a 128-byte boundary of shared memory (TMA destinations)
    float2* bufs = reinterpret_cast<float2*>(smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127));
    float2* tws = bufs + X::BUFS * X::BUF;
    using Job = YJob<X, INV>;
    const int nxb = ceil_div(g.Mxp, Job::TX), nzb = ceil_div(g.nz, Job::NP);
    Job job{W, tws, &tmap, bh, g.nz, g.Mxp, g.Ky, g.My, nxb, nzb, nxb * nzb * ncomp, (size_t)X::N * g.Mxp};
    X::table(tws, tw);
    col_loop<X>(bufs, state, tma, err, job);
}

template <class X, bool INV>
cudaError_t launch(float2* W, const Geom& g, const double2* tw, int ncomp, const StepState* st, const CUtensorMap& map,
                   int bh, int* err, cudaStream_t s)
{
    constexpr int TX = kTX, NP = X::C / TX;
    const long long tiles = (long long)ceil_div(g.Mxp, TX) * ceil_div(g.nz, NP) * ncomp;
    k_ycol<X, INV><<<col_grid<X>(k_ycol<X, INV>, tiles), X::THREADS, X::kSmem, s>>>(W, g, tw, ncomp, st, map, bh, err,
                                                                                    current_batch().mb);
    return cudaGetLastError();
}

}  // namespace

int ycol_full(int ny)
{
    switch (ny) {
#define FLUSI_CASE(n, R, L) case n: return y_cols<n>();
        FLUSI_COL_LENGTHS(FLUSI_CASE)
#undef FLUSI_CASE
    default: return 0;
    }
}

cudaError_t launch_ycol(bool inverse, int cols, float2* W, const Geom& g, const double2* tw, int ncomp, const StepState* st,
                        const CUtensorMap& map, int bh, int* err, cudaStream_t s)
{
    switch (g.ny) {
#define FLUSI_CASE(n, R, L)                                                                                  \
    case n:                                                                                                  \
        if (cols == y_cols<n>())                                                                             \
            return inverse ? launch<Col<R, L, y_cols<n>()>, true>(W, g, tw, ncomp, st, map, bh, err, s)       \
                           : launch<Col<R, L, y_cols<n>()>, false>(W, g, tw, ncomp, st, map, bh, err, s);     \
        return inverse ? launch<Col<R, L, kTX>, true>(W, g, tw, ncomp, st, map, bh, err, s)                   \
                       : launch<Col<R, L, kTX>, false>(W, g, tw, ncomp, st, map, bh, err, s);
        FLUSI_COL_LENGTHS(FLUSI_CASE)
#undef FLUSI_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t configure_ycol(int ny)
{
    cudaError_t e = cudaSuccess;
    auto one = [&](const void* kernel, size_t smem) {
        if (!e) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
#define FLUSI_KERNELS(X)                                       \
    one((const void*)k_ycol<X, true>, X::kSmem);               \
    one((const void*)k_ycol<X, false>, X::kSmem);
    switch (ny) {
#define FLUSI_CASE(n, R, L)                                    \
    case n: {                                                  \
        using Full = Col<R, L, y_cols<n>()>;                   \
        using Small = Col<R, L, kTX>;                          \
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
