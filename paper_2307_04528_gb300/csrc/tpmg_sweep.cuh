// Block-Jacobi sweeps of Eq. (1) with the column solve split over segments
// of layers.
//
// Both recurrences of the column solve are first-order and linear, so a
// segment of layers acts on the value entering it as an affine map.  With
// the setup factors m = 1/p and f = t/p, p = q + t, the forward elimination
//   y_k = (v_k + t_{k-1} y_{k-1}) m_k
// is carried as h_k = t_k y_k = f_k w_k, w_k = v_k + h_{k-1}, y_k = m_k w_k:
// t_z is not read at all (20 -> 16 bytes per cell from a zero guess in FP32, 32
// -> 28 on a guess).  f is kept as g (LevelDev): where q is the smaller part of
// the pivot, w - (q/p) w keeps the row sums that a rounded f would lose, where t
// is, f w keeps the coupling that 1 - q/p would lose.  The backward substitution
// x_k = y_k + f_k x_{k+1} is as in the serial sweep (smooth_column); the maps of
// both directions share the factor A = prod f.
//
// A thread owns CV adjacent columns and LZ consecutive layers; QL lanes sit
// side by side along longitude, so a warp covers QL CV columns of 32 / QL
// segments and a block all segments of those columns.  Every load of the sweep
// is independent of the recurrences: a thread issues them all at once, where
// a thread walking a column keeps a few layers in flight, and the segments'
// maps are then exchanged through shared memory, each thread combining the
// maps below (above) its own to the value entering its segment before it
// re-runs its layers with the serial formulas.  Each array is read once.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "tpmg_device.cuh"
#include "tpmg_internal.h"

namespace tpmg {

// CV adjacent values of T, loaded and stored together.
template <typename T, int CV>
struct Vals {
    T a[CV];
};

template <typename T, int CV>
struct VecOf;
template <>
struct VecOf<float, 2> {
    using type = float2;
};
template <>
struct VecOf<float, 4> {
    using type = float4;
};
template <>
struct VecOf<double, 2> {
    using type = double2;
};

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> ldv(const T *__restrict__ p, unsigned byte)
{
    Vals<T, CV> r;
    const char *q = reinterpret_cast<const char *>(p) + byte;
    if constexpr (CV == 1) {
        r.a[0] = __ldg(reinterpret_cast<const T *>(q));
    } else {
        using V = typename VecOf<T, CV>::type;
        const V v = __ldg(reinterpret_cast<const V *>(q));
        r.a[0] = v.x;
        r.a[1] = v.y;
        if constexpr (CV == 4) {
            r.a[2] = v.z;
            r.a[3] = v.w;
        }
    }
    return r;
}

// The same of a vector that the kernel before this one may have written
// (after_previous) or that this one writes: not through the read-only path.
template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> ldv_of(const T *p, unsigned byte)
{
    Vals<T, CV> r;
    const char *q = reinterpret_cast<const char *>(p) + byte;
    if constexpr (CV == 1) {
        r.a[0] = *reinterpret_cast<const T *>(q);
    } else {
        using V = typename VecOf<T, CV>::type;
        const V v = *reinterpret_cast<const V *>(q);
        r.a[0] = v.x;
        r.a[1] = v.y;
        if constexpr (CV == 4) {
            r.a[2] = v.z;
            r.a[3] = v.w;
        }
    }
    return r;
}

template <typename T, int CV>
__device__ __forceinline__ void stv(T *__restrict__ p, unsigned byte, const Vals<T, CV> &x)
{
    char *q = reinterpret_cast<char *>(p) + byte;
    if constexpr (CV == 1) {
        *reinterpret_cast<T *>(q) = x.a[0];
    } else {
        using V = typename VecOf<T, CV>::type;
        V v;
        v.x = x.a[0];
        v.y = x.a[1];
        if constexpr (CV == 4) {
            v.z = x.a[2];
            v.w = x.a[3];
        }
        *reinterpret_cast<V *>(q) = v;
    }
}

// Element-wise arithmetic; two FP32 values per instruction (f32x2).
__device__ __forceinline__ unsigned long long pk(float x, float y)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void upk(unsigned long long r, float &x, float &y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(r));
}

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> vfma(const Vals<T, CV> &x, const Vals<T, CV> &y,
                                            const Vals<T, CV> &z)
{
    Vals<T, CV> r;
    if constexpr (sizeof(T) == 4 && CV % 2 == 0) {
#pragma unroll
        for (int i = 0; i < CV; i += 2) {
            unsigned long long d;
            asm("fma.rn.f32x2 %0, %1, %2, %3;"
                : "=l"(d)
                : "l"(pk(x.a[i], x.a[i + 1])), "l"(pk(y.a[i], y.a[i + 1])),
                  "l"(pk(z.a[i], z.a[i + 1])));
            upk(d, r.a[i], r.a[i + 1]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < CV; ++i) r.a[i] = fma(x.a[i], y.a[i], z.a[i]);
    }
    return r;
}

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> vadd(const Vals<T, CV> &x, const Vals<T, CV> &y)
{
    Vals<T, CV> r;
    if constexpr (sizeof(T) == 4 && CV % 2 == 0) {
#pragma unroll
        for (int i = 0; i < CV; i += 2) {
            unsigned long long d;
            asm("add.rn.f32x2 %0, %1, %2;"
                : "=l"(d)
                : "l"(pk(x.a[i], x.a[i + 1])), "l"(pk(y.a[i], y.a[i + 1])));
            upk(d, r.a[i], r.a[i + 1]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < CV; ++i) r.a[i] = x.a[i] + y.a[i];
    }
    return r;
}

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> vmul(const Vals<T, CV> &x, const Vals<T, CV> &y)
{
    Vals<T, CV> r;
    if constexpr (sizeof(T) == 4 && CV % 2 == 0) {
#pragma unroll
        for (int i = 0; i < CV; i += 2) {
            unsigned long long d;
            asm("mul.rn.f32x2 %0, %1, %2;"
                : "=l"(d)
                : "l"(pk(x.a[i], x.a[i + 1])), "l"(pk(y.a[i], y.a[i + 1])));
            upk(d, r.a[i], r.a[i + 1]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < CV; ++i) r.a[i] = x.a[i] * y.a[i];
    }
    return r;
}

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> splat(T x)
{
    Vals<T, CV> r;
#pragma unroll
    for (int i = 0; i < CV; ++i) r.a[i] = x;
    return r;
}

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> vneg(const Vals<T, CV> &x)
{
    if constexpr (sizeof(T) == 4 && CV % 2 == 0) {  // two per instruction
        return vmul<T, CV>(x, splat<T, CV>(T(-1)));
    } else {
        Vals<T, CV> r;
#pragma unroll
        for (int i = 0; i < CV; ++i) r.a[i] = -x.a[i];
        return r;
    }
}

template <typename T, int CV>
__device__ __forceinline__ Vals<T, CV> lds_v(const T *p)
{
    Vals<T, CV> r;
    if constexpr (CV == 1) {
        r.a[0] = *p;
    } else {
        using V = typename VecOf<T, CV>::type;
        const V v = *reinterpret_cast<const V *>(p);
        r.a[0] = v.x;
        r.a[1] = v.y;
        if constexpr (CV == 4) {
            r.a[2] = v.z;
            r.a[3] = v.w;
        }
    }
    return r;
}

// How the link factors f, kept as g (LevelDev), are taken:
//   LINK_LESS_ONE  every g of the level is f - 1: f w = g w + w.  The coarse levels of a
//                  lat-lon grid, bound by latency: a cluster solve of 8 x 6 x 70 19.6 us
//                  instead of 21.7, the FP32 V-cycle of 88 x 60 x 70 58.8 instead of 60.3
//   LINK_EITHER    w counts where g is f - 1: in FP64 by a select, in FP32 by a factor
//                  of one or zero.  The finest levels, at whose poles the horizontal
//                  couplings outweigh the vertical ones (1 to 4 % of the warps; a vote
//                  of the warp for the short form undid the order of the loads: with
//                  <b, u_out> at 512 x 384 x 70 in FP32 84 -> 150 us)
//   LINK_DIRECTED  g = -q/p, with f = d m (the coupling down of the row above times
//                  1/p) beside it
enum { LINK_LESS_ONE, LINK_EITHER, LINK_DIRECTED };

// One where g is f - 1, else zero: a saturated product, which issues on the FMA pipe
// (selects by g's sign go to the integer pipe at half its rate; the FP32 V-cycle at
// 1024 x 768 x 70: 1.11 -> 1.03 ms); no negative g lies above -2^-126
// (launch_column_lu).  volatile: formed anew at each use instead of held in registers.
__device__ __forceinline__ float one_of(float g)
{
    float z;
    asm volatile("mul.rn.sat.f32 %0, %1, %2;" : "=f"(z) : "f"(g), "f"(-0x1p127f));
    return z;
}
template <int CV>
__device__ __forceinline__ Vals<float, CV> vone(const Vals<float, CV> &g)
{
    Vals<float, CV> r;
#pragma unroll
    for (int i = 0; i < CV; ++i) r.a[i] = one_of(g.a[i]);
    return r;
}

// f w, w = v + h.  In FP32 the w that counts is formed beside w, as z h + z v, so
// that the chain from h to f w stays two operations long.
template <int LINK, typename T, int CV>
__device__ __forceinline__ Vals<T, CV> carry(const Vals<T, CV> &g, const Vals<T, CV> &f,
                                             const Vals<T, CV> &v, const Vals<T, CV> &h,
                                             const Vals<T, CV> &w)
{
    if constexpr (LINK == LINK_DIRECTED) {
        return vmul<T, CV>(f, w);
    } else if constexpr (LINK == LINK_LESS_ONE) {
        return vfma<T, CV>(g, w, w);
    } else if constexpr (sizeof(T) == 4) {
        const Vals<T, CV> z = vone(g);
        return vfma<T, CV>(g, w, vfma<T, CV>(z, h, vmul<T, CV>(z, v)));
    } else {
        Vals<T, CV> r;
#pragma unroll
        for (int i = 0; i < CV; ++i) r.a[i] = fma(g.a[i], w.a[i], whole(g.a[i], w.a[i]));
        return r;
    }
}

// y + f x; in a directed level x + (y - (q/p) x).
template <int LINK, typename T, int CV>
__device__ __forceinline__ Vals<T, CV> back(const Vals<T, CV> &g, const Vals<T, CV> &x,
                                            const Vals<T, CV> &y)
{
    const Vals<T, CV> t = vfma<T, CV>(g, x, y);
    if constexpr (LINK != LINK_EITHER) {
        return vadd<T, CV>(x, t);
    } else if constexpr (sizeof(T) == 4) {
        return vfma<T, CV>(vone(g), x, t);
    } else {
        Vals<T, CV> r;
#pragma unroll
        for (int i = 0; i < CV; ++i) r.a[i] = whole(g.a[i], x.a[i]) + t.a[i];
        return r;
    }
}

// A Chebyshev step instead of a sweep: with b the residual and u_in the step d,
// r_out = b - H d, x += d (first: x = d) and u_out = c1 d + c2 H_z^{-1} r_out;
// last: x takes the new step too.  Each cell of x is its own thread's.
template <typename T>
struct ChebStep {
    T *r_out, *x;
    T c1, c2;
    bool first, last;
};

// One tile of QL CV columns.  DOT: returns the thread's part of <b, u_out>,
// b waiting for the last pass in the thread's own slots of shared memory.
// Byte offsets are 32-bit (pick).  sh: 3 blockDim CV values (4 in a directed
// level), and LZ blockDim CV more for DOT.
template <typename T, int CV, int LZ, int QL, bool GUESS, bool DOT, int LINK, bool CHEB = false,
          typename Level>
__device__ __forceinline__ T sweep_tile(const Level &L, const T *b, const T *uin,
                                        T *__restrict__ uout, T omega, int tile, T *sh,
                                        const ChebStep<T> &ch = {})
{
    using X = Vals<T, CV>;
    constexpr unsigned SZ = sizeof(T);
    constexpr bool NS = kDirected<Level>;
    static_assert(NS == (LINK == LINK_DIRECTED), "a level's own link form");
    static_assert(!(NS && DOT), "no <b, u_out> of a directed level");
    const int nlon = L.nlon, nlat = L.nlat, nz = L.nz;
    const int ncol = nlon * nlat;
    const int q = threadIdx.x % QL, seg = threadIdx.x / QL, nseg = blockDim.x / QL;
    const int own = (tile * QL + q) * CV;
    const int col = own < ncol ? own : ncol - CV;  // past the end: read, not stored
    const int k0 = seg * LZ;
    const unsigned plane = (unsigned)ncol * SZ;
    const unsigned first = (unsigned)col * SZ + (unsigned)min(k0, nz - 1) * plane;
    const int row = blockDim.x * CV;  // values per slot row of shared memory
    T *sb = sh + 3 * row + threadIdx.x * CV;

    X v[LZ], m[LZ], g[LZ], uc[GUESS ? LZ : 1], f[NS ? LZ : 1];
    // No load sits behind a branch: layers past the top re-read the last one.
    unsigned off = first;
#pragma unroll
    for (int c = 0; c < LZ; ++c) {
        m[c] = ldv<T, CV>(L.m, off);
        g[c] = ldv<T, CV>(factor_of(L), off);
        v[c] = ldv_of<T, CV>(b, off);
        if (GUESS) uc[c] = ldv_of<T, CV>(uin, off);
        if constexpr (NS) f[c] = ldv<T, CV>(down_of(L), off);
        off += k0 + c + 1 < nz ? plane : 0u;
    }
    if (GUESS) {
        const int j = col / nlon, i = col - j * nlon;
        const bool hasN = j + 1 < nlat, hasS = j > 0;
        // rows past a pole read the cell itself
        const T *ue = uin + (i + CV == nlon ? -i : CV), *uw = uin + (i == 0 ? nlon - 1 : -1);
        const T *un = uin + (hasN ? nlon : 0), *us = uin - (hasS ? nlon : 0);
        const T *tw = west_of(L) + (i == 0 ? nlon - 1 : -1);
        const T *ts = south_of(L) - (hasS ? nlon : 0);
        off = first;
        // CHEB: t_z and d of the layer below the segment, d of the one above (a
        // segment past the top has none: with one layer there is none to read)
        X tzd = splat<T, CV>(T(0)), ud = tzd, ua = tzd;
        if constexpr (CHEB) {
            const unsigned dn = k0 > 0 && k0 < nz ? plane : 0u;
            tzd = ldv<T, CV>(up_of(L), first - dn);
            ud = ldv_of<T, CV>(uin, first - dn);
            ua = ldv_of<T, CV>(uin, first + (k0 + LZ < nz ? LZ * plane : 0u));
        }
#pragma unroll
        for (int c = 0; c < LZ; ++c) {
            const X t = ldv<T, CV>(east_of(L), off);
            X tb = t;  // the couplings of the cells to the west
            if constexpr (NS && CV > 1) tb = ldv<T, CV>(west_of(L), off);
            const X N = ldv_of<T, CV>(un, off), S = ldv_of<T, CV>(us, off);
            const X tn = ldv<T, CV>(north_of(L), off), tS = ldv<T, CV>(ts, off);
            const T E = ldv_of<T, 1>(ue, off).a[0], W = ldv_of<T, 1>(uw, off).a[0];
            const T tW = ldv<T, 1>(tw, off).a[0];
            if constexpr (CHEB) {
                // r = b - H d in flux form
                const X hm = ldv<T, CV>(mass_of(L), off), tz = ldv<T, CV>(up_of(L), off);
                const X &U = c + 1 < LZ ? uc[c + 1 < LZ ? c + 1 : c] : ua;
                const X &D = c > 0 ? uc[c > 0 ? c - 1 : 0] : ud;
#pragma unroll
                for (int e = 0; e < CV; ++e) {
                    const T x = uc[c].a[e];
                    T s = hm.a[e] * x;
                    s = fma(t.a[e], x - (e + 1 < CV ? uc[c].a[e + 1 < CV ? e + 1 : e] : E), s);
                    s = fma(e > 0 ? t.a[e > 0 ? e - 1 : 0] : tW,
                            x - (e > 0 ? uc[c].a[e > 0 ? e - 1 : 0] : W), s);
                    if (hasN) s = fma(tn.a[e], x - N.a[e], s);
                    if (hasS) s = fma(tS.a[e], x - S.a[e], s);
                    if (k0 + c + 1 < nz) s = fma(tz.a[e], x - U.a[e], s);
                    if (k0 + c > 0) s = fma(tzd.a[e], x - D.a[e], s);
                    v[c].a[e] -= s;
                }
                tzd = tz;
                off += k0 + c + 1 < nz ? plane : 0u;
                continue;
            }
            if (DOT) stv<T, CV>(sb + c * row, 0u, v[c]);
#pragma unroll
            for (int e = 0; e < CV; ++e) {
                v[c].a[e] = fma(t.a[e], e + 1 < CV ? uc[c].a[e + 1 < CV ? e + 1 : e] : E, v[c].a[e]);
                v[c].a[e] = fma(e > 0 ? tb.a[e > 0 ? e - 1 : 0] : tW,
                                e > 0 ? uc[c].a[e > 0 ? e - 1 : 0] : W, v[c].a[e]);
            }
            const X vn = vfma<T, CV>(tn, N, v[c]);
            v[c] = hasN ? vn : v[c];
            const X vs = vfma<T, CV>(tS, S, v[c]);
            v[c] = hasS ? vs : v[c];
            off += k0 + c + 1 < nz ? plane : 0u;
        }
        if constexpr (CHEB) {  // behind every load, which the compiler keeps in order with it
            off = first;
#pragma unroll
            for (int c = 0; c < LZ; ++c, off += plane)
                if (own < ncol && k0 + c < nz) stv<T, CV>(ch.r_out, off, v[c]);
        }
    }
    // layers past the top: 1/p = 0 makes their y and x zero; a directed level's
    // q/p takes the sign of its uses
    const X zero = splat<T, CV>(T(0));
#pragma unroll
    for (int c = 0; c < LZ; ++c) {
        m[c] = k0 + c < nz ? m[c] : zero;
        if constexpr (NS) {
            g[c] = vneg<T, CV>(g[c]);
            f[c] = vmul<T, CV>(f[c], m[c]);
        }
    }

    // forward: the segment's map h_out = A h_in + C; backward factor B (= A in
    // a symmetric level)
    X A = splat<T, CV>(T(1)), C = zero, B = A;
#pragma unroll
    for (int c = 0; c < LZ; ++c) {
        const X t = vadd<T, CV>(v[c], C);
        C = carry<LINK, T, CV>(g[c], f[NS ? c : 0], v[c], C, t);
        A = carry<LINK, T, CV>(g[c], f[NS ? c : 0], zero, A, A);
        if (NS) B = vfma<T, CV>(g[c], B, B);
    }
    T *sA = sh + q * CV, *sC = sA + row, *sF = sC + row, *sB = sA;
    if constexpr (NS) {
        sB = sh + (3 + (DOT ? LZ : 0)) * row + q * CV;
        stv<T, CV>(sB + seg * QL * CV, 0u, B);
    }
    stv<T, CV>(sA + seg * QL * CV, 0u, A);
    stv<T, CV>(sC + seg * QL * CV, 0u, C);
    __syncthreads();
    X h = zero;
    for (int s = 0; s < seg; ++s)
        h = vfma<T, CV>(lds_v<T, CV>(sA + s * QL * CV), h, lds_v<T, CV>(sC + s * QL * CV));
    // the segment's layers with the value entering it; v now holds y.  F:
    // the backward map x_bottom = A x_above + F
#pragma unroll
    for (int c = 0; c < LZ; ++c) {
        const X w = vadd<T, CV>(v[c], h);
        h = carry<LINK, T, CV>(g[c], f[NS ? c : 0], v[c], h, w);
        v[c] = vmul<T, CV>(w, m[c]);
    }
    X xv[CHEB ? LZ : 1];
    if constexpr (CHEB) {
        off = first;
#pragma unroll
        for (int c = 0; c < LZ; ++c) {
            xv[c] = ch.first ? zero : ldv_of<T, CV>(ch.x, off);
            off += k0 + c + 1 < nz ? plane : 0u;
        }
    }
    X F = zero;
#pragma unroll
    for (int c = LZ - 1; c >= 0; --c) F = back<LINK, T, CV>(g[c], F, v[c]);
    stv<T, CV>(sF + seg * QL * CV, 0u, F);
    __syncthreads();
    X x = zero;
    for (int s = nseg - 1; s > seg; --s)
        x = vfma<T, CV>(lds_v<T, CV>(sB + s * QL * CV), x, lds_v<T, CV>(sF + s * QL * CV));
    const X om = splat<T, CV>(omega), om1 = splat<T, CV>(T(1) - omega);
    T acc = 0;
    off = first + (unsigned)(min(LZ, nz - k0) - 1) * plane;
#pragma unroll
    for (int c = LZ - 1; c >= 0; --c) {
        x = back<LINK, T, CV>(g[c], x, v[c]);
        X uo;
        if constexpr (CHEB) {
            uo = vfma<T, CV>(splat<T, CV>(ch.c2), x, vmul<T, CV>(splat<T, CV>(ch.c1), uc[c]));
            xv[c] = vadd<T, CV>(xv[c], uc[c]);
            if (ch.last) xv[c] = vadd<T, CV>(xv[c], uo);
        } else {
            uo = vmul<T, CV>(om, x);
            if (GUESS) uo = vfma<T, CV>(om1, uc[c], uo);
        }
        if (k0 + c < nz) {
            if (own < ncol) {
                if constexpr (CHEB) stv<T, CV>(ch.x, off, xv[c]);
                stv<T, CV>(uout, off, uo);
                if (DOT) {
                    const X bc = lds_v<T, CV>(sb + c * row);
#pragma unroll
                    for (int e = 0; e < CV; ++e) acc = fma(bc.a[e], uo.a[e], acc);
                }
            }
            off -= plane;
        }
    }
    return acc;
}

// The coarsest-level solve (`sweeps` sweeps from zero) by one thread-block
// cluster: block r owns the latitude rows [r R, r R + R), and a thread (column,
// segment of LZ layers) of them keeps its factors, couplings and right-hand
// side in registers for all sweeps.  u lives in the blocks' shared memory, two
// copies written in turn; the rows beside a block's own are read from its
// neighbours' shared memory, and one cluster barrier separates the sweeps.
// The forward and backward maps of the segments are exchanged as in
// sweep_tile, their factors once.  sh: 2 R nlon nz + 4 blockDim values.
template <typename T, int LZ, int LINK, typename Level>
__device__ __forceinline__ void coarse_cluster(const Level &L, const T *b,
                                               T *__restrict__ out, T omega, int sweeps, int R,
                                               T *sh)
{
    namespace cg = cooperative_groups;
    constexpr bool NS = kDirected<Level>;
    cg::cluster_group cl = cg::this_cluster();
    const int nlon = L.nlon, nlat = L.nlat, nz = L.nz, plane = nlon * nlat;
    const int rank = (int)cl.block_rank(), j0 = rank * R;
    const int rows = max(0, min(R, nlat - j0)), cols = rows * nlon, part = R * nlon;
    T *u0 = sh, *u1 = sh + part * nz;
    T *sA = sh + 2 * part * nz, *sC = sA + blockDim.x, *sF = sC + blockDim.x;
    T *sB = NS ? sF + blockDim.x : sA;
    const int nseg = (nz + LZ - 1) / LZ;
    const bool mine = (int)threadIdx.x < cols * nseg;
    const int seg = mine ? threadIdx.x / cols : 0, lc = mine ? threadIdx.x - seg * cols : 0;
    const int k0 = seg * LZ;
    const int r = lc / nlon, i = lc - r * nlon, j = min(j0 + r, nlat - 1);
    const int de = (i + 1 == nlon) ? -i : 1, dw = (i == 0) ? nlon - 1 : -1;
    const bool hasN = j + 1 < nlat, hasS = j > 0;
    // the cells north and south of this column's first layer, in both copies
    const T *n0 = u0 + lc, *s0 = u0 + lc;
    if (hasN)
        n0 = r + 1 < rows ? u0 + lc + nlon : cl.map_shared_rank(u0, rank + 1) + i;
    if (hasS)
        s0 = r > 0 ? u0 + lc - nlon : cl.map_shared_rank(u0, rank - 1) + (R - 1) * nlon + i;
    using X = Vals<T, 1>;
    T m[LZ], bb[LZ], te[LZ], tw[LZ], tn[LZ], ts[LZ], uc[LZ];
    X g[LZ], f[NS ? LZ : 1];
#pragma unroll
    for (int c = 0; c < LZ; ++c) {
        const int o = min(k0 + c, nz - 1) * plane + j * nlon + i;
        bb[c] = b[o];
        te[c] = __ldg(east_of(L) + o);
        tw[c] = __ldg(west_of(L) + o + dw);
        tn[c] = hasN ? __ldg(north_of(L) + o) : T(0);
        ts[c] = hasS ? __ldg(south_of(L) + o - nlon) : T(0);
        m[c] = k0 + c < nz ? __ldg(L.m + o) : T(0);
        g[c].a[0] = NS ? -__ldg(factor_of(L) + o) : __ldg(factor_of(L) + o);
        uc[c] = 0;
        if constexpr (NS) f[c].a[0] = __ldg(down_of(L) + o) * m[c];
    }
    const X zero = {{T(0)}};
    X A = {{T(1)}}, B = A;
#pragma unroll
    for (int c = 0; c < LZ; ++c) {
        A = carry<LINK, T, 1>(g[c], f[NS ? c : 0], zero, A, A);
        if (NS) B = vfma<T, 1>(g[c], B, B);
    }
    sA[threadIdx.x] = A.a[0];
    if (NS) sB[threadIdx.x] = B.a[0];
    const T om1 = T(1) - omega;
    for (int it = 0; it < sweeps; ++it) {
        const int cur = (it & 1) * part * nz;  // the copy read; the other is written
        T *nxt = (it & 1) ? u0 : u1;
        X v[LZ], C = zero;
#pragma unroll
        for (int c = 0; c < LZ; ++c) {
            T x = bb[c];
            if (it > 0) {
                const int o = cur + min(k0 + c, nz - 1) * part;
                x = fma(te[c], u0[o + lc + de], x);
                x = fma(tw[c], u0[o + lc + dw], x);
                x = fma(tn[c], n0[o], x);
                x = fma(ts[c], s0[o], x);
            }
            v[c].a[0] = x;
        }
#pragma unroll
        for (int c = 0; c < LZ; ++c)
            C = carry<LINK, T, 1>(g[c], f[NS ? c : 0], v[c], C, vadd<T, 1>(v[c], C));
        sC[threadIdx.x] = C.a[0];
        __syncthreads();
        X h = zero;
#pragma unroll 4
        for (int s = 0; s < seg; ++s) h.a[0] = fma(sA[s * cols + lc], h.a[0], sC[s * cols + lc]);
        X F = zero;
#pragma unroll
        for (int c = 0; c < LZ; ++c) {
            const X w = vadd<T, 1>(v[c], h);
            h = carry<LINK, T, 1>(g[c], f[NS ? c : 0], v[c], h, w);
            v[c].a[0] = w.a[0] * m[c];
        }
#pragma unroll
        for (int c = LZ - 1; c >= 0; --c) F = back<LINK, T, 1>(g[c], F, v[c]);
        sF[threadIdx.x] = F.a[0];
        __syncthreads();
        X x = zero;
#pragma unroll 4
        for (int s = nseg - 1; s > seg; --s)
            x.a[0] = fma(sB[s * cols + lc], x.a[0], sF[s * cols + lc]);
#pragma unroll
        for (int c = LZ - 1; c >= 0; --c) v[c] = x = back<LINK, T, 1>(g[c], x, v[c]);
#pragma unroll
        for (int c = LZ - 1; c >= 0; --c) {
            uc[c] = fma(om1, uc[c], omega * v[c].a[0]);
            if (mine && k0 + c < nz) {
                if (it + 1 < sweeps)
                    nxt[(k0 + c) * part + lc] = uc[c];
                else
                    out[(k0 + c) * plane + j * nlon + i] = uc[c];
            }
        }
        cl.sync();  // the sweep is complete, in every block, before the next reads it
    }
}

}  // namespace tpmg
