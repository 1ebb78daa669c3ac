// Launchers of the segmented sweeps (tpmg_sweep.cuh) and of the coarsest-level
// solve on a thread-block cluster, and the rules that pick a shape for a level.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "tpmg_internal.h"
#include "tpmg_sweep.cuh"

namespace tpmg {
namespace {

// A block takes the tiles blockIdx, + gridDim, ...: one, unless a level has
// more tiles than there are slots for partial sums.  (The loop also has the
// compiler issue a tile's loads in one run: 0.534 ms against 0.698 without it
// at 1536 x 1152 x 70, the same instructions otherwise, on q/p alone.)
template <typename T, int CV, int LZ, int QL, bool GUESS, bool DOT, int LINK, int MAXT, int MINB,
          typename Level>
__global__ void __launch_bounds__(MAXT, MINB)
k_sweep(Level L, const T *b, const T *uin, T *__restrict__ uout, T omega,
        double *__restrict__ partial, const int *flag)
{
    after_previous();
    if (flag && !*flag) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tiles = (L.nlon * L.nlat + QL * CV - 1) / (QL * CV);
    T acc = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (tile != (int)blockIdx.x) __syncthreads();  // the last tile's maps have been read
        acc += sweep_tile<T, CV, LZ, QL, GUESS, DOT, LINK>(L, b, uin, uout, omega, tile,
                                                           reinterpret_cast<T *>(smraw));
    }
    if (DOT) block_store<0>((double)acc, partial);
}

// A Chebyshev step of the coarsest-level solve as one sweep (launch_cheb_sweep).
template <typename T, int CV, int LZ, int QL, int LINK, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
k_sweep_cheb(LevelDev<T> L, const T *b, const T *uin, T *__restrict__ uout, ChebStep<T> ch)
{
    after_previous();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tiles = (L.nlon * L.nlat + QL * CV - 1) / (QL * CV);
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (tile != (int)blockIdx.x) __syncthreads();  // the last tile's maps have been read
        sweep_tile<T, CV, LZ, QL, true, false, LINK, true>(L, b, uin, uout, T(1), tile,
                                                           reinterpret_cast<T *>(smraw), ch);
    }
}

// A shape of the sweep: CV columns per thread, LZ layers per segment, QL
// lanes along longitude, MAXT threads at most, MINB blocks per SM.
template <int CV_, int LZ_, int QL_, int MAXT_, int MINB_, bool GUESS_ = true>
struct Shape {
    static constexpr int CV = CV_, LZ = LZ_, QL = QL_, MAXT = MAXT_, MINB = MINB_;
    static constexpr bool GUESS = GUESS_;  // false: sweeps from zero only
};

// FP32 levels that fill the GPU.  From zero the sweep reads b, 1/p and g and is
// bound by HBM: pairs of columns in 256-byte rows (1536 x 1152 x 70: 0.480 ->
// 0.278 ms, 7.1 TB/s; quads and single columns, on q/p alone, 0.290 and 0.316
// against 0.274).  On a guess a thread also reads five arrays around it, and
// instructions bind beside HBM: quads of columns (16-byte loads), 64 columns to
// a block of 128 threads so that two blocks share an SM (0.777 -> 0.560 ms, 6.2
// TB/s; with <b, u_out> 0.817 -> 0.653; on q/p alone 0.534 and 0.627, one block
// of 256 threads 0.584 and 0.659, pairs 0.77 and 1.04).
using Large0 = Shape<2, 9, 32, 256, 3, false>;
using Large = Shape<4, 9, 16, 128, 2>;
// the same with segments of 5 layers, for layer counts that leave fewer of
// their slots empty (256 x 192 x 50: 10.7 -> 9.2 us; 352 x 226 x 37: 17.1 -> 11.7)
using Large5 = Shape<4, 5, 16, 256, 2>;
// rows that are no multiple of 2 columns (only from zero: 0.316 ms as above)
using Odd0 = Shape<1, 9, 32, 256, 4, false>;
// Levels of 2048 to 8192 columns in FP32: latency; 32 columns to a block
// (48 x 82 x 70 on a guess: 13.5 -> 3.2 us, Large 3.6)
using Mid = Shape<2, 5, 16, 256, 2>;
// Small levels: 8 columns to a block, short segments (24 x 46 x 70 on a guess:
// FP32 4.7 -> 2.8 us, Mid 3.2; 8 x 18 x 70 in FP64: 43 -> 6.2 us)
using Small = Shape<1, 3, 8, 192, 1>;
using SmallTall = Shape<1, 3, 8, 512, 1>;  // more than 72 layers
// FP64 levels from 2^16 cells to 8192 columns, where the extra FP64 operations
// of the exchanged maps begin to count: long segments (64 x 98 x 70 on a guess:
// 43.8 -> 21.2 us, Small 26.2; 64 x 32 x 16: 9.6 -> 7.6, Small 4.4)
using Mid64 = Shape<1, 9, 8, 192, 1>;

// Directed FP32 levels that fill the GPU: one more array per layer in
// registers, two more read around it, so segments of 5 layers for the quads
// and 2 blocks per SM from zero.  All sweeps of a V-cycle of H and one of H^T
// at 512 x 384 x 70, column walks against these and the smaller shapes: 1.66
// -> 0.50 ms, the coarsest level's 2 x 12 included.
using NsLarge0 = Shape<2, 9, 32, 256, 2, false>;
using NsLarge = Shape<4, 5, 16, 256, 2>;

// f(LINK_*) for the form of a level's link factors.
template <typename Level, typename F>
auto with_link(const Level &L, F &&f)
{
    if constexpr (kDirected<Level>) {
        return f(std::integral_constant<int, LINK_DIRECTED>{});
    } else {
        return L.either ? f(std::integral_constant<int, LINK_EITHER>{})
                        : f(std::integral_constant<int, LINK_LESS_ONE>{});
    }
}

template <typename T, typename S, bool GUESS, bool DOT, int LINK, typename Level = LevelDev<T>>
constexpr auto kernel_of()
{
    return k_sweep<T, S::CV, S::LZ, S::QL, GUESS, DOT, LINK, S::MAXT, S::MINB, Level>;
}

template <typename S>
int threads_of(int nz)  // whole warps: a segment past the last owns no layer
{
    return ((nz + S::LZ - 1) / S::LZ * S::QL + 31) / 32 * 32;
}

template <typename T, typename S, bool DOT, typename Level = LevelDev<T>>
constexpr size_t smem_of(int threads)
{
    return (size_t)(3 + kDirected<Level> + (DOT ? S::LZ : 0)) * threads * S::CV * sizeof(T);
}

template <typename T, typename S, typename Level>
bool suits(const Level &L, uintptr_t ptrs)
{
    return L.nlon % S::CV == 0 && threads_of<S>(L.nz) <= S::MAXT && ptrs % (S::CV * sizeof(T)) == 0;
}

// The arguments of one sweep; count: only its number of blocks is wanted.
template <typename T>
struct Sweep {
    const T *b, *uin;
    T *uout;
    double omega;
    double *partial;
    cudaStream_t s;
    const int *flag;
    bool dot, count;
    const ChebStep<T> *ch = nullptr;  // a Chebyshev step
};

template <typename T, typename S, typename Level>
int go(const Level &L, const Sweep<T> &a)
{
    const long long per = S::QL * S::CV;
    const long long tiles = ((long long)L.nlon * L.nlat + per - 1) / per;
    const int grid = (int)std::min<long long>(tiles, kReduceSlots), threads = threads_of<S>(L.nz);
    static_assert(smem_of<T, S, S::GUESS, Level>(S::MAXT) <= 48 * 1024, "no opt-in is asked for");
    if (a.count) return grid;
    const T *b = a.b, *uin = a.uin;
    T *uout = a.uout;
    double *partial = a.partial;
    const double omega = a.omega;
    const cudaStream_t s = a.s;
    const int *flag = a.flag;
    with_link(L, [&](auto link) {
        constexpr int LINK = decltype(link)::value;
        if (!uin)
            launch_after(kernel_of<T, S, false, false, LINK, Level>(), grid, threads,
                         smem_of<T, S, false, Level>(threads), s, L, b, uin, uout, (T)omega,
                         partial, flag);
        if constexpr (S::GUESS && !kDirected<Level>) {
            if (a.ch) {
                launch_after(k_sweep_cheb<T, S::CV, S::LZ, S::QL, LINK, S::MAXT, S::MINB>, grid,
                             threads, smem_of<T, S, false>(threads), s, L, b, uin, uout, *a.ch);
                return;
            }
        }
        if constexpr (S::GUESS) {
            if constexpr (!kDirected<Level>)
                if (uin && partial)
                    launch_after(kernel_of<T, S, true, true, LINK>(), grid, threads,
                                 smem_of<T, S, true>(threads), s, L, b, uin, uout, (T)omega,
                                 partial, flag);
            if (uin && !partial)
                launch_after(kernel_of<T, S, true, false, LINK, Level>(), grid, threads,
                             smem_of<T, S, false, Level>(threads), s, L, b, uin, uout, (T)omega,
                             partial, flag);
        }
    });
    return grid;
}

// Slots left empty by segments of lz layers, in percent of the layers.
int waste(int nz, int lz) { return ((nz + lz - 1) / lz * lz - nz) * 100 / nz; }

constexpr int kSmallColumns = 2048, kMidColumns = 8192;

constexpr int kClusterBlocks = 8;  // the portable cluster size

// Threads of a block of the coarsest-level solve: what its registers allow.
template <typename T, int LZ, typename Level>
constexpr int kClusterThreads = sizeof(T) == 4 && !kDirected<Level> ? 512
                                : sizeof(T) == 4 || LZ <= 4         ? 384
                                                                    : 256;

template <typename T, int LZ, int LINK, typename Level>
__global__ void __launch_bounds__(kClusterThreads<T, LZ, Level>, 1)
k_coarse_cluster(Level L, const T *b, T *__restrict__ out, T omega, int sweeps, int R)
{
    after_previous();
    extern __shared__ __align__(16) unsigned char smraw[];
    coarse_cluster<T, LZ, LINK, Level>(L, b, out, omega, sweeps, R, reinterpret_cast<T *>(smraw));
}

// Layers per segment, balancing the dependent steps: about ten operations a
// layer against two a segment, plus in FP32 (4 clocks an operation, FP64 ten
// times that) the reads of the exchange.
template <typename T>
int cluster_lz(int nz)
{
    if (sizeof(T) == 8) return nz <= 24 ? 2 : nz <= 48 ? 3 : nz <= 96 ? 4 : 6;
    return nz <= 16 ? 4 : nz <= 40 ? 6 : nz <= 72 ? 8 : 12;
}

struct ClusterShape {
    int lz, R, blocks, threads;
    size_t values;  // of shared memory
};

template <typename T>
ClusterShape cluster_shape(int nlon, int nlat, int nz)
{
    ClusterShape c;
    c.lz = cluster_lz<T>(nz);
    // at least 128 cells to a block
    const int blocks = (int)std::min<long long>(
        kClusterBlocks, std::max<long long>((long long)nlon * nlat * nz / 128, 1));
    c.R = (nlat + blocks - 1) / blocks;
    c.blocks = (nlat + c.R - 1) / c.R;
    c.threads = (c.R * nlon * ((nz + c.lz - 1) / c.lz) + 31) / 32 * 32;
    c.values = 2 * (size_t)c.R * nlon * nz + 4 * (size_t)c.threads;
    return c;
}

// Layers a block of shape S holds for nz, its empty slots and segments included.
template <typename S>
int slots_of(int nz)
{
    return threads_of<S>(nz) / S::QL * S::LZ;
}

// Whether an FP64 level of at most 8192 columns sweeps by segments (slots: of the long
// segments, 0: of the short ones) rather than by the column walk.  The walk takes its
// serial chain, some 1.8 + 0.25 nz us from zero and 1.7 + 0.61 nz on a guess whatever
// the columns; the segments their FP64 operations, empty slots included, about 3.5 +
// 2.1e-5 us a slot from zero (3e-5 beyond 800,000) and 5 + 4.4e-5 on a guess.  In us,
// segments and walk: 128 x 64 x 16 from zero 8.1 and 5.8, on a guess 11.4 and 9.7;
// x 70 15.0 and 19.3, 25.0 and 43.0; x 76 26.4 and 20.7, 39 and 47; 64 x 98 x 50 12.9
// and 14.3, 20.9 and 31.2.  A Chebyshev step is weighed against the walk, the residual
// by cells and the vector update (7 of them, 96 x 80 x 50: 292 and 236 us; x 70: 294
// and 306).
bool fp64_segments(long long ncol, int nz, int slots, bool guess, bool cheb)
{
    if (slots == 0) return cheb || nz > 4;  // 32 x 32 x 4: 3.1 and 2.7 us, x 6 3.1 and 3.4
    const double s = (double)ncol * slots;
    if (cheb) return 6.0 * s < 2.5e5 + 2.5e4 * nz + 2.7 * (double)ncol * nz;
    if (guess) return s < 13900.0 * nz - 75000.0;
    return s < std::min(12000.0 * nz - 80000.0, 8200.0 * nz + 52000.0);
}

// The shape for a level and its buffers, or -1 where the column walk is the
// faster form: FP64 levels beyond 8192 columns (the maps cost 16 FP64
// operations per cell against 10, and the walk is bound by the FP64 pipe) or of
// few layers (fp64_segments), FP32 levels that fill the GPU with rows of no
// whole quad, and layer counts beyond the shapes' threads (FP32 levels that fill
// the GPU: 72, or 75 by segments of 5).
template <typename T, typename Level>
int pick(const Level &L, const Sweep<T> &a)
{
    const long long ncol = (long long)L.nlon * L.nlat;
    if ((unsigned long long)ncol * L.nz * sizeof(T) >= 1ull << 32) return -1;  // 32-bit offsets
    const uintptr_t ptrs = (uintptr_t)a.b | (uintptr_t)a.uin | (uintptr_t)a.uout |
                           (uintptr_t)east_of(L) | (uintptr_t)north_of(L) |
                           (uintptr_t)west_of(L) | (uintptr_t)south_of(L) |
                           (uintptr_t)down_of(L) | (uintptr_t)L.m | (uintptr_t)factor_of(L) |
                           (uintptr_t)mass_of(L) | (uintptr_t)up_of(L) |
                           (a.ch ? (uintptr_t)a.ch->r_out | (uintptr_t)a.ch->x : 0);
    if constexpr (sizeof(T) == 8) {
        if (ncol > kMidColumns) return -1;
        const bool mid = ncol * L.nz >= 1 << 16 && suits<T, Mid64>(L, ptrs);
        if constexpr (!kDirected<Level>)
            if (!fp64_segments(ncol, L.nz, mid ? slots_of<Mid64>(L.nz) : 0, a.uin != nullptr,
                               a.ch != nullptr))
                return -1;
        if (mid) return go<T, Mid64>(L, a);
    } else if (ncol < kMidColumns) {
        if (ncol >= kSmallColumns && suits<T, Mid>(L, ptrs)) return go<T, Mid>(L, a);
    } else if constexpr (kDirected<Level>) {
        if (a.uin) return suits<T, NsLarge>(L, ptrs) ? go<T, NsLarge>(L, a) : -1;
        return suits<T, NsLarge0>(L, ptrs) ? go<T, NsLarge0>(L, a) : -1;
    } else {
        if (waste(L.nz, 9) >= waste(L.nz, 5) + 8 && suits<T, Large5>(L, ptrs))
            return go<T, Large5>(L, a);
        if (a.uin || a.dot) return suits<T, Large>(L, ptrs) ? go<T, Large>(L, a) : -1;
        if (suits<T, Large0>(L, ptrs)) return go<T, Large0>(L, a);
        return suits<T, Odd0>(L, ptrs) ? go<T, Odd0>(L, a) : -1;
    }
    return suits<T, Small>(L, ptrs) ? go<T, Small>(L, a) : go<T, SmallTall>(L, a);
}

}  // namespace

template <typename T>
int launch_sweep(const LevelDev<T> &L, const T *b, const T *uin, T *uout, double omega,
                 double *partial, cudaStream_t s, const int *flag)
{
    return pick<T>(L, {b, uin, uout, omega, partial, s, flag, partial != nullptr, false});
}

template <typename T>
bool cheb_sweep_fits(const LevelDev<T> &L, const T *b, const T *d, T *d_out, T *r_out, T *x)
{
    const ChebStep<T> ch{r_out, x, T(0), T(0), false, false};
    return pick<T>(L, {b, d, d_out, 1.0, nullptr, nullptr, nullptr, false, true, &ch}) >= 0;
}

template <typename T>
cudaError_t launch_cheb_sweep(const LevelDev<T> &L, const T *b, const T *d, T *d_out, T *r_out,
                              T *x, double c1, double c2, bool first, bool last, cudaStream_t s)
{
    const ChebStep<T> ch{r_out, x, (T)c1, (T)c2, first, last};
    pick<T>(L, {b, d, d_out, 1.0, nullptr, s, nullptr, false, false, &ch});
    return cudaGetLastError();
}

template <typename T>
int smooth_dot_partials(const LevelDev<T> &L, const T *b, const T *uin, T *uout)
{
    const int n = pick<T>(L, {b, uin, uout, 0.0, nullptr, nullptr, nullptr, true, true});
    return n >= 0 ? n : (L.nlon * L.nlat + kBlock - 1) / kBlock;
}

// Levels whose rows fit eight blocks' threads take the cluster (up to 448
// columns of 70 layers in FP32, 168 in FP64).  Per sweep, FP32: 1.35 us at 11
// x 18 x 37 and 1.8 us at 6 x 14 x 70, against 4.5 and 4.1 us for one block
// with the level's factors in registers and ~3 us for a launch per sweep.
template <typename T>
bool coarse_solve_fits(int nlon, int nlat, int nz)
{
    if (nlon > 512) return false;
    const ClusterShape c = cluster_shape<T>(nlon, nlat, nz);
    const int most = c.lz <= 4 ? kClusterThreads<T, 4, LevelDev<T>>
                               : kClusterThreads<T, 6, LevelDev<T>>;
    return c.threads <= most && c.values * sizeof(T) <= 160 * 1024;
}

template <typename T>
bool ns_coarse_fits(const NsView<T> &V)
{
    if (V.nlon > 512) return false;
    const ClusterShape c = cluster_shape<T>(V.nlon, V.nlat, V.nz);
    const int most = c.lz <= 4 ? kClusterThreads<T, 4, NsView<T>>
                               : kClusterThreads<T, 6, NsView<T>>;
    return c.threads <= most && c.values * sizeof(T) <= 160 * 1024;
}

template <typename T, typename Level>
static cudaError_t coarse_solve(const Level &L, const T *b, T *out, double omega, int sweeps,
                                cudaStream_t s)
{
    const ClusterShape c = cluster_shape<T>(L.nlon, L.nlat, L.nz);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c.blocks);
    cfg.blockDim = dim3(c.threads);
    cfg.dynamicSmemBytes = c.values * sizeof(T);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c.blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1] = after_attribute();
    cfg.attrs = at;
    cfg.numAttrs = capturing(s) ? 1 : 2;
    const T om = (T)omega;
    auto run = [&](auto lz) {
        return with_link(L, [&](auto link) {
            return cudaLaunchKernelEx(
                &cfg, k_coarse_cluster<T, decltype(lz)::value, decltype(link)::value, Level>, L, b,
                out, om, sweeps, c.R);
        });
    };
    if constexpr (sizeof(T) == 8) {
        if (c.lz == 2) return run(std::integral_constant<int, 2>{});
        if (c.lz == 3) return run(std::integral_constant<int, 3>{});
        if (c.lz == 4) return run(std::integral_constant<int, 4>{});
        return run(std::integral_constant<int, 6>{});
    } else {
        if (c.lz == 4) return run(std::integral_constant<int, 4>{});
        if (c.lz == 6) return run(std::integral_constant<int, 6>{});
        if (c.lz == 8) return run(std::integral_constant<int, 8>{});
        return run(std::integral_constant<int, 12>{});
    }
}

template <typename T>
cudaError_t launch_coarse_solve(const LevelDev<T> &L, const T *b, T *out, double omega, int sweeps,
                                cudaStream_t s)
{
    return coarse_solve<T>(L, b, out, omega, sweeps, s);
}

template <typename T>
cudaError_t launch_ns_coarse(const NsView<T> &V, const T *b, T *out, double omega, int sweeps,
                             cudaStream_t s)
{
    return coarse_solve<T>(V, b, out, omega, sweeps, s);
}

template <typename T>
int launch_ns_sweep(const NsView<T> &V, const T *b, const T *u_in, T *u_out, double omega,
                    cudaStream_t s)
{
    return pick<T>(V, {b, u_in, u_out, omega, nullptr, s, nullptr, false, false});
}

template <typename T, typename Level, int... LINK>
static cudaError_t allow_coarse_smem()
{
    constexpr int A = sizeof(T) == 4 ? 8 : 2, B = sizeof(T) == 4 ? 12 : 3;
    for (const void *k : {(const void *)k_coarse_cluster<T, 4, LINK, Level>...,
                          (const void *)k_coarse_cluster<T, 6, LINK, Level>...,
                          (const void *)k_coarse_cluster<T, A, LINK, Level>...,
                          (const void *)k_coarse_cluster<T, B, LINK, Level>...}) {
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t sweep_prepare()
{
    for (cudaError_t q :
         {allow_coarse_smem<float, LevelDev<float>, LINK_EITHER, LINK_LESS_ONE>(),
          allow_coarse_smem<double, LevelDev<double>, LINK_EITHER, LINK_LESS_ONE>(),
          allow_coarse_smem<float, NsView<float>, LINK_DIRECTED>(),
          allow_coarse_smem<double, NsView<double>, LINK_DIRECTED>()})
        if (q != cudaSuccess) return q;
    return cudaSuccess;
}

#define TPMG_SWEEP_INST(T)                                                                       \
    template int launch_sweep<T>(const LevelDev<T> &, const T *, const T *, T *, double, double *, \
                                 cudaStream_t, const int *);                                     \
    template bool cheb_sweep_fits<T>(const LevelDev<T> &, const T *, const T *, T *, T *, T *);    \
    template cudaError_t launch_cheb_sweep<T>(const LevelDev<T> &, const T *, const T *, T *, T *, \
                                              T *, double, double, bool, bool, cudaStream_t);     \
    template int smooth_dot_partials<T>(const LevelDev<T> &, const T *, const T *, T *);           \
    template bool coarse_solve_fits<T>(int, int, int);                                             \
    template cudaError_t launch_coarse_solve<T>(const LevelDev<T> &, const T *, T *, double, int, \
                                                cudaStream_t);                                    \
    template int launch_ns_sweep<T>(const NsView<T> &, const T *, const T *, T *, double,          \
                                    cudaStream_t);                                                \
    template bool ns_coarse_fits<T>(const NsView<T> &);                                            \
    template cudaError_t launch_ns_coarse<T>(const NsView<T> &, const T *, T *, double, int,       \
                                             cudaStream_t);
TPMG_SWEEP_INST(double)
TPMG_SWEEP_INST(float)
#undef TPMG_SWEEP_INST

}  // namespace tpmg
