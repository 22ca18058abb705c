// Transforms of tile columns in two register passes, for the FP32 y and z passes
// at lengths n = R L that are worth a kernel of their own: C columns of n rows in
// shared memory, row-major, as a TMA box lands them.
//
// Pass 1 takes a column's rows j + L t, t < R, per thread (radix R, the twiddles
// w_n^{j q}, back in place); pass 2 the rows q L + i, i < L (radix L), whose
// outputs are the frequencies q + R i, straight to global memory.  A tile thus
// crosses shared memory three times (read, write, read) and meets one block
// barrier between, where a plan of three radix-8 stages crosses it five times
// with two; every offset is a compile-time constant.  Of an inverse transform's
// rows those that the 2/3 rule drops are neither loaded nor cleared: pass 1 takes
// zero for them.
//
// The kernels are persistent: a block keeps its twiddle table and loops over
// tiles, and as soon as pass 2 has read a tile the next one's copies go out into
// its place.  Loads, not arithmetic, are what these passes wait for.
//   Radices up to 18 run three blocks of 256 threads per SM, one tile each, at 80
//   registers a thread: the y and forward z passes fit but for 24 bytes of spills
//   at 324 rows; the inverse z pass, which holds side rows besides, spills 148 and
//   128 bytes at 324 rows (8 and 16 columns), 56 and 120 at 288, 80 and 20 at 256
//   (8 and 32), up to 28 at 162 to 216.  Two blocks per SM were not measured for it.
//   Larger ones leave two groups of 256 threads, but shared memory for three
//   tiles: they form one block of two groups over a ring of three tiles, each
//   group taking every second load, so that one tile is always on its way (y
//   inverse at 512^3: 0.68 ms as two blocks of one tile, 0.56 so).
//   Over 512 rows a 64 KB tile would have 8 columns, 64-byte rows that share
//   128-byte lines with a neighbour's: such tiles in a ring took 8.4 ms for the y
//   inverse at 1024^3, as two blocks 5.4 to 6.3, in the z inverse 7.8.  There a
//   block of 512 threads takes 16 columns, 128 KB in two halves of the rows over a
//   ring of three halves (the first half of the next tile flies while this one
//   is transformed): 5.1 and 4.3 ms, the forward passes 2.3 and 1.7 (z staged 2.8).

// A tile's rows are C consecutive values, so a warp's 8-byte accesses cover whole
// 128-byte lines (C >= 16); with C = 8 (the narrow z tile, up to 512 rows) pass 2
// meets each bank twice.
#pragma once

#include "fft.cuh"
#include "kernels.cuh"

namespace flusi {
namespace {

// columns of a full tile of length n (64 KB of shared memory; over 512 rows 16
// columns), at most `most`
constexpr int col_tile(int n, int most)
{
    int c = 8;
    while (2 * c * n <= (n > 512 ? 16384 : 8192) && 2 * c <= most) c *= 2;
    return c;
}

template <int R_, int L_, int C_> struct Col {
    static constexpr int R = R_, L = L_, C = C_, N = R * L;
    static constexpr int CH = N > 512 ? 2 : 1;                 // loads (row ranges) of a tile
    static constexpr int T = CH == 2 ? 512 : 256;              // threads of a group
    static constexpr int U1 = L * C, U2 = R * C;               // threads' work items of the passes
    static constexpr int ROUNDS1 = (U1 + T - 1) / T, ROUNDS2 = (U2 + T - 1) / T;
    static constexpr bool SMALL = R <= 18 && L <= 18;
    static constexpr int GROUPS = SMALL || CH == 2 ? 1 : 2, BUFS = SMALL ? 1 : 3;
    static constexpr int THREADS = GROUPS * T, MINB = SMALL ? 3 : 1;
    // values of a buffer: a row range, up to the next 128-byte boundary, where the
    // next buffer's TMA boxes land (243 rows of 8 columns end 64 bytes short of one)
    static constexpr int BUF = (N * C / CH + 15) / 16 * 16;
    static constexpr size_t kSmem = sizeof(float2) * ((size_t)BUFS * BUF + N) + 128;
    static_assert((C & (C - 1)) == 0 && BUF <= 8192 && (CH == 1 || (R % 2 == 0 && !SMALL)), "a tile");
    static_assert(BUFS == 1 || BUF * sizeof(float2) % 128 == 0, "TMA destinations");

    // A tile: the buffer of its rows, or of its first and its second half of rows.
    struct Tile {
        float2 *lo, *hi;
        // row range q of L rows (q < R)
        __device__ __forceinline__ float2* rows(int q) const
        {
            if constexpr (CH == 1) return lo + q * L * C;
            else return q < R / 2 ? lo + q * L * C : hi + (q - R / 2) * L * C;
        }
    };

    // rows [lo, hi] of a transform that keeps |m| <= K, K = N/3 or (strict rule,
    // N divisible by 3) N/3 - 1: 0 all dropped, 2 all kept, 1 it depends
    __host__ __device__ static constexpr int kept(int lo, int hi)
    {
        constexpr int most = N / 3, least = N % 3 == 0 ? N / 3 - 1 : N / 3;
        if (hi <= least || lo >= N - least) return 2;
        if (lo > most && hi < N - most) return 0;
        return 1;
    }

    __device__ __forceinline__ static void table(float2* tws, const double2* tw)
    {
        const float2* w = reinterpret_cast<const float2*>(tw + N);   // the FP32 copy
        for (int i = threadIdx.x; i < N; i += THREADS) tws[i] = w[(i / L) * (i % L)];   // w_n^{q j} at q L + j
    }

    // pass 1; PRUNED: rows of dropped modes are zero (whatever the tile holds
    // there); weigh(v, row) may scale an input
    template <bool INV, bool PRUNED, class Weigh>
    __device__ __forceinline__ static void first(const Tile& tile, const float2* tws, int tid, int K, Weigh weigh)
    {
#pragma unroll 1
        for (int rd = 0; rd < ROUNDS1; ++rd) {
            const int u = tid + rd * T;
            if (U1 % T != 0 && u >= U1) break;
            const int j = u / C;
            float2 v[R];                              // rows j + L t of column u % C
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int k = PRUNED ? kept(L * t, L * t + L - 1) : 2;
                const int row = j + L * t;
                if (k == 0) v[t] = make_float2(0.0f, 0.0f);
                else if (k == 2) v[t] = weigh(tile.rows(t)[u], row);
                else v[t] = row <= K || row >= N - K ? weigh(tile.rows(t)[u], row) : make_float2(0.0f, 0.0f);
            }
            Dft<float, R, INV>::run(v);
            tile.rows(0)[u] = v[0];
#pragma unroll
            for (int q = 1; q < R; ++q) {
                float2 w = tws[q * L + j];
                if (INV) w.y = -w.y;
                tile.rows(q)[u] = cmul(v[q], w);
            }
        }
    }

    // pass 2: io.begin(q, col) before a work item's values are read, io.all(a)
    // with a[i] the value of frequency q + R i; refill() once every value is
    // read.  Every thread of the group calls it.
    template <bool INV, class Io, class Refill>
    __device__ __forceinline__ static void second(const Tile& tile, int tid, Io& io, Refill refill)
    {
#pragma unroll 1
        for (int rd = 0; rd < ROUNDS2; ++rd) {
            const int u = tid + rd * T;
            const bool on = U2 % T == 0 || u < U2;
            const int q = u / C, col = u % C;
            float2 a[L];
            if (on) {
                io.begin(q, col);
                const float2* p = tile.rows(q) + col;
#pragma unroll
                for (int i = 0; i < L; ++i) a[i] = p[i * C];
            }
            if (rd == ROUNDS2 - 1) refill();
            if (on) {
                Dft<float, L, INV>::run(a);
                io.all(a);
            }
        }
    }
};

// barriers of one group of threads: all of it meets, or the first warp waits
// for the others (who do not wait).  Ids 1 and 2 for group 0, 3 and 4 for group 1.
template <int T> __device__ __forceinline__ void group_sync(int group)
{
    if (group == 0) asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
    else asm volatile("bar.sync 3, %0;" ::"n"(T) : "memory");
}
template <int T> __device__ __forceinline__ void group_gather(int group)
{
    if (group == 0) asm volatile("bar.sync 2, %0;" ::"n"(T) : "memory");
    else asm volatile("bar.sync 4, %0;" ::"n"(T) : "memory");
}
template <int T> __device__ __forceinline__ void group_report(int group)
{
    if (group == 0) asm volatile("bar.arrive 2, %0;" ::"n"(T) : "memory");
    else asm volatile("bar.arrive 4, %0;" ::"n"(T) : "memory");
}

struct ColState {
    unsigned long long full[3];   // per buffer: its load has landed
    int issued[3];                // per buffer: loads sent so far
    int bad[2];                   // per group: a wait gave up
};

// The tiles of a block, numbered 0, 1, 2, ...: tile i belongs to group i % GROUPS
// and takes the loads i CH + h, h < CH (its row ranges).  Load s lands in buffer
// s % BUFS, as that buffer's load number s / BUFS.
// Job: bool exists(i) (false from some i on), issue(i, h, buf, bar) by one thread
// (TMA boxes, after an expect_tx) or copy(i, h, buf, tid) by a group's threads
// (16-byte copies), work(i, tile, tid, group, refill).
//
// A buffer's barrier tells two loads apart only by parity, so a group first
// waits until its load has been sent (the one before it in that buffer has then
// landed and been read), then for the landing; both waits are bounded.  A group
// that gives up reports FLUSI_ETIMEOUT and leaves its loop; what it no longer
// sends lets the other one's wait run out too, and the block then waits (bounded)
// for every TMA load in flight, and each thread for its own copies, before it ends.
// limit: of a wait, in SM clocks (as mbar_wait).
template <class X, class Job>
__device__ __forceinline__ void col_loop(float2* bufs, ColState& sh, bool tma, int* err, Job& job,
                                         const long long limit = 400000000LL)
{
    constexpr int CH = X::CH;
    const int group = X::GROUPS == 1 ? 0 : (threadIdx.x >= X::T ? 1 : 0), tid = threadIdx.x & (X::T - 1);
    auto slot_of = [](int s) { return X::BUFS == 1 ? 0 : s % X::BUFS; };
    auto buffer = [&](int s) { return bufs + slot_of(s) * X::BUF; };
    auto sent = [&](int s) { *(volatile int*)&sh.issued[slot_of(s)] = s / X::BUFS + 1; };
    auto send = [&](int s) {      // one thread
        job.issue(s / CH, s % CH, buffer(s), sh.full + slot_of(s));
        sent(s);
    };
    auto copy_in = [&](int s) {   // the group's threads; each arrives when its copies have landed
        job.copy(s / CH, s % CH, buffer(s), tid);
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(sh.full + slot_of(s)))
                     : "memory");
        if (tid == 0) sent(s);
    };
    if (threadIdx.x == 0) {
        for (int b = 0; b < X::BUFS; ++b) {
            mbar_init(sh.full + b, tma ? 1 : X::T);
            sh.issued[b] = 0;
        }
        sh.bad[0] = sh.bad[1] = 0;
    }
    __syncthreads();   // the state (and the caller's tables) are set
    if (tma) {
        if (threadIdx.x == 0)
            for (int s = 0; s < X::BUFS; ++s)
                if (job.exists(s / CH)) send(s);
    } else if (group == 0) {
        for (int s = 0; s < X::BUFS; ++s)
            if (job.exists(s / CH)) copy_in(s);
    }
#pragma unroll 1
    for (int i = group; job.exists(i); i += X::GROUPS) {
        bool ok = true;
#pragma unroll
        for (int h = 0; h < CH; ++h) {
            const int s = i * CH + h, load = s / X::BUFS;
            const long long t0 = clock64();
            while (ok && *(volatile int*)&sh.issued[slot_of(s)] <= load) ok = clock64() - t0 <= limit;
            if (ok) ok = mbar_wait(sh.full + slot_of(s), (unsigned)load & 1u, limit);
        }
        if (!ok) {
            *(volatile int*)&sh.bad[group] = 1;
            atomicCAS(err, 0, (int)FLUSI_ETIMEOUT);
        }
        __syncwarp();
        group_sync<X::T>(group);
        if (*(volatile int*)&sh.bad[group]) break;   // only this group sets it, before the barrier
        const int next = i * CH + X::BUFS;
        typename X::Tile tile{buffer(i * CH), buffer(i * CH + CH - 1)};
        job.work(i, tile, tid, group, [&] {
            // the group has read the tile: refill its buffers
            if (!job.exists(next / CH)) return;
            if (!tma) {
                group_sync<X::T>(group);
                for (int h = 0; h < CH; ++h)
                    if (job.exists((next + h) / CH)) copy_in(next + h);
            } else if (tid < 32) {
                group_gather<X::T>(group);
                if (tid == 0) {
                    fence_proxy_async();   // the generic accesses to the tile before the asynchronous proxy's
                    for (int h = 0; h < CH; ++h)
                        if (job.exists((next + h) / CH)) send(next + h);
                }
                __syncwarp();
            } else {
                group_report<X::T>(group);
            }
        });
    }
    if (!tma) cp_async_wait_all();
    __syncthreads();
    if (tma && threadIdx.x == 0 && (sh.bad[0] | sh.bad[1]))
        for (int b = 0; b < X::BUFS; ++b)
            if (sh.issued[b] > 0) mbar_wait(sh.full + b, (unsigned)(sh.issued[b] - 1) & 1u, limit);
}

// The lengths served, X(n, R, L): from 64 rows on all but 729 (the halves of a tile
// over 512 rows need an even R) and 972 (no R, L up to 32).  Those, tiles narrowed
// by y_cols or z_cols, the other plans and FP64 take the staged kernels of ypass.cu
// and zpass.cu.
#define FLUSI_COL_LENGTHS(X)                                                                               \
    X(64, 8, 8) X(72, 9, 8) X(81, 9, 9) X(96, 12, 8) X(108, 12, 9) X(128, 16, 8) X(144, 12, 12)            \
    X(162, 18, 9) X(192, 16, 12) X(216, 18, 12) X(243, 27, 9) X(256, 16, 16) X(288, 18, 16) X(324, 18, 18) \
    X(384, 24, 16) X(432, 27, 16) X(486, 27, 18) X(512, 32, 16) X(576, 24, 24) X(648, 24, 27)              \
    X(768, 32, 24) X(864, 32, 27) X(1024, 32, 32)

// Persistent grid of a kernel with `smem` bytes over `tiles` tiles per member.
template <class X, class K> dim3 col_grid(K kernel, long long tiles)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, X::THREADS, X::kSmem);
    const long long n = current_batch().n, resident = (long long)sm_count() * (per_sm > 0 ? per_sm : 1);
    const long long share = (resident + n - 1) / n;
    return dim3((unsigned)(tiles < share ? tiles : share), 1, (unsigned)n);
}

}  // namespace
}  // namespace flusi
