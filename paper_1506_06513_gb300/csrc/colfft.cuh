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
// its place.  Loads, not arithmetic, are what these passes wait for.  Radices up
// to 18 leave registers for three blocks of 256 threads per SM, one tile each.
// Larger ones leave two groups of 256 threads, but shared memory for three
// tiles: they form one block of two groups over a ring of three tiles, each
// group taking every second load, so that one tile is always on its way (y
// inverse at 512^3: 0.68 ms as two blocks of one tile, 0.56 so).  Tiles of 8
// columns stay two blocks of one tile: their 64-byte rows share 128-byte lines
// with a neighbour's, and more of them in flight cost more than the overlap gives
// (y inverse at 1024^3: 5.4 ms, 8.4 in the ring).

// A tile's rows are C consecutive values, so a warp's 8-byte accesses cover whole
// 128-byte lines (C >= 16); with C = 8 (n > 512) pass 2 meets each bank twice.
#pragma once

#include "fft.cuh"
#include "kernels.cuh"

namespace flusi {
namespace {

constexpr int kColThreads = 256;   // of a group

// columns of a full tile (64 KB of shared memory) of length n, at most `most`
constexpr int col_tile(int n, int most)
{
    int c = 8;
    while (2 * c * n <= 8192 && 2 * c <= most) c *= 2;
    return c;
}

template <int R_, int L_, int C_> struct Col {
    static constexpr int R = R_, L = L_, C = C_, N = R * L, T = kColThreads;
    static constexpr int U1 = L * C, U2 = R * C;               // threads' work items of the passes
    static constexpr int ROUNDS1 = (U1 + T - 1) / T, ROUNDS2 = (U2 + T - 1) / T;
    static constexpr bool SMALL = R <= 18 && L <= 18;
    static constexpr int GROUPS = SMALL || C == 8 ? 1 : 2, BUFS = GROUPS == 1 ? 1 : 3;
    static constexpr int THREADS = GROUPS * T, MINB = GROUPS == 2 ? 1 : SMALL ? 3 : 2;
    static constexpr size_t kSmem = sizeof(float2) * ((size_t)BUFS * N * C + N) + 128;
    static_assert((C & (C - 1)) == 0 && N * C <= 8192, "a tile");

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
    __device__ __forceinline__ static void first(float2* buf, const float2* tws, int tid, int K, Weigh weigh)
    {
#pragma unroll 1
        for (int rd = 0; rd < ROUNDS1; ++rd) {
            const int u = tid + rd * T;
            if (U1 % T != 0 && u >= U1) break;
            const int j = u / C;
            float2* p = buf + u;                      // row j, column u % C
            float2 v[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int k = PRUNED ? kept(L * t, L * t + L - 1) : 2;
                const int row = j + L * t;
                if (k == 0) v[t] = make_float2(0.0f, 0.0f);
                else if (k == 2) v[t] = weigh(p[t * L * C], row);
                else v[t] = row <= K || row >= N - K ? weigh(p[t * L * C], row) : make_float2(0.0f, 0.0f);
            }
            Dft<float, R, INV>::run(v);
            p[0] = v[0];
#pragma unroll
            for (int q = 1; q < R; ++q) {
                float2 w = tws[q * L + j];
                if (INV) w.y = -w.y;
                p[q * L * C] = cmul(v[q], w);
            }
        }
    }

    // pass 2: io.begin(q, col) before a work item's values are read, io.all(a)
    // with a[i] the value of frequency q + R i; refill() once every value is
    // read.  Every thread of the group calls it.
    template <bool INV, class Io, class Refill>
    __device__ __forceinline__ static void second(const float2* buf, int tid, Io& io, Refill refill)
    {
#pragma unroll 1
        for (int rd = 0; rd < ROUNDS2; ++rd) {
            const int u = tid + rd * T;
            const bool on = U2 % T == 0 || u < U2;
            const int q = u / C, col = u % C;
            float2 a[L];
            if (on) {
                io.begin(q, col);
                const float2* p = buf + q * L * C + col;
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
__device__ __forceinline__ void group_sync(int group)
{
    if (group == 0) asm volatile("bar.sync 1, %0;" ::"n"(kColThreads) : "memory");
    else asm volatile("bar.sync 3, %0;" ::"n"(kColThreads) : "memory");
}
__device__ __forceinline__ void group_gather(int group)
{
    if (group == 0) asm volatile("bar.sync 2, %0;" ::"n"(kColThreads) : "memory");
    else asm volatile("bar.sync 4, %0;" ::"n"(kColThreads) : "memory");
}
__device__ __forceinline__ void group_report(int group)
{
    if (group == 0) asm volatile("bar.arrive 2, %0;" ::"n"(kColThreads) : "memory");
    else asm volatile("bar.arrive 4, %0;" ::"n"(kColThreads) : "memory");
}

struct ColState {
    unsigned long long full[3];   // per buffer: its load has landed
    int issued[3];                // per buffer: loads sent so far
    int bad[2];                   // per group: a wait gave up
};

// The loads of a block, numbered 0, 1, 2, ...: load i lands in buffer i % BUFS,
// as that buffer's load number i / BUFS, and belongs to group i % GROUPS.
// Job: bool exists(i) (false from some i on), issue(i, buf, bar) by one thread
// (TMA boxes, after an expect_tx) or copy(i, buf, tid) by a group's threads
// (16-byte copies), work(i, buf, tid, group, refill).
//
// A buffer's barrier tells two loads apart only by parity, so a group first
// waits until its load has been sent (the one before it in that buffer has then
// landed and been read), then for the landing; both waits are bounded.  A group
// that gives up reports FLUSI_ETIMEOUT and leaves its loop; what it no longer
// sends lets the other one's wait run out too, and the block then waits (bounded)
// for every load in flight before it ends.
template <class X, class Job>
__device__ __forceinline__ void col_loop(float2* bufs, ColState& sh, bool tma, int* err, Job& job)
{
    constexpr long long kLimit = 400000000LL;   // SM clocks, as mbar_wait
    const int group = X::GROUPS == 1 ? 0 : (threadIdx.x >= X::T ? 1 : 0), tid = threadIdx.x & (X::T - 1);
    auto slot_of = [](int i) { return X::BUFS == 1 ? 0 : i % X::BUFS; };
    auto buffer = [&](int i) { return bufs + slot_of(i) * (X::N * X::C); };
    auto sent = [&](int i) { *(volatile int*)&sh.issued[slot_of(i)] = i / X::BUFS + 1; };
    auto send = [&](int i) {      // one thread
        job.issue(i, buffer(i), sh.full + slot_of(i));
        sent(i);
    };
    auto copy_in = [&](int i) {   // the group's threads; each arrives when its copies have landed
        job.copy(i, buffer(i), tid);
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(sh.full + slot_of(i)))
                     : "memory");
        if (tid == 0) sent(i);
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
            for (int i = 0; i < X::BUFS; ++i)
                if (job.exists(i)) send(i);
    } else if (group == 0) {
        for (int i = 0; i < X::BUFS; ++i)
            if (job.exists(i)) copy_in(i);
    }
#pragma unroll 1
    for (int i = group; job.exists(i); i += X::GROUPS) {
        const int load = i / X::BUFS;
        bool ok = true;
        const long long t0 = clock64();
        while (ok && *(volatile int*)&sh.issued[slot_of(i)] <= load) ok = clock64() - t0 <= kLimit;
        if (ok) ok = mbar_wait(sh.full + slot_of(i), (unsigned)load & 1u, kLimit);
        if (!ok) {
            *(volatile int*)&sh.bad[group] = 1;
            atomicCAS(err, 0, (int)FLUSI_ETIMEOUT);
        }
        __syncwarp();
        group_sync(group);
        if (*(volatile int*)&sh.bad[group]) break;   // only this group sets it, before the barrier
        const int next = i + X::BUFS;
        job.work(i, buffer(i), tid, group, [&] {
            // the group has read the tile: refill it
            if (!job.exists(next)) return;
            if (!tma) {
                group_sync(group);
                copy_in(next);
            } else if (tid < 32) {
                group_gather(group);
                if (tid == 0) {
                    fence_proxy_async();   // the generic accesses to the tile before the asynchronous proxy's
                    send(next);
                }
                __syncwarp();
            } else {
                group_report(group);
            }
        });
    }
    __syncthreads();
    if (tma && threadIdx.x == 0 && (sh.bad[0] | sh.bad[1]))
        for (int b = 0; b < X::BUFS; ++b)
            if (sh.issued[b] > 0) mbar_wait(sh.full + b, (unsigned)(sh.issued[b] - 1) & 1u, kLimit);
}

// The lengths served, X(n, R, L).  Others (and narrowed tiles, the other plans
// and FP64) take the staged kernels of ypass.cu and zpass.cu, and so do the z
// passes over 512: with 8 columns a tile the two-pass inverse is slower there
// (1024^3: 7.8 ms against 6.5, its side rows need more registers than are left).
#define FLUSI_COL_SHORT(X)                                                                                 \
    X(64, 8, 8) X(72, 9, 8) X(81, 9, 9) X(96, 12, 8) X(108, 12, 9) X(128, 16, 8) X(144, 12, 12)            \
    X(162, 18, 9) X(192, 16, 12) X(216, 18, 12) X(243, 27, 9) X(256, 16, 16) X(288, 18, 16) X(324, 18, 18) \
    X(384, 24, 16) X(432, 27, 16) X(486, 27, 18) X(512, 32, 16)
#define FLUSI_COL_LENGTHS(X) \
    FLUSI_COL_SHORT(X) X(576, 24, 24) X(648, 27, 24) X(768, 32, 24) X(864, 32, 27) X(1024, 32, 32)

inline int col_sms()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}
// Persistent grid of a kernel with `smem` bytes over `tiles` tiles per member.
template <class X, class K> dim3 col_grid(K kernel, long long tiles)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, X::THREADS, X::kSmem);
    const long long n = current_batch().n, resident = (long long)col_sms() * (per_sm > 0 ? per_sm : 1);
    const long long share = (resident + n - 1) / n;
    return dim3((unsigned)(tiles < share ? tiles : share), 1, (unsigned)n);
}

}  // namespace
}  // namespace flusi
