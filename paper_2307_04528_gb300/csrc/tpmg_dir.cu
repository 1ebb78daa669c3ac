// The FP32 direction update + apply of the conjugate-gradient iteration (q = H
// d, d = z + beta d_old, <d, q>) with a thread per four adjacent columns
// walking a range of layers.
//
// Every own-cell array is read and written as 16-byte vectors: 11 vector and 5
// scalar loads for four cells, where the column walk (dir_apply_column)
// issues 16 loads a cell, and the layers are split between blocks until the
// GPU is full.  Every value enters the arithmetic in the operation and order
// of the column walk, so d and q are equal bit for bit; the partial sums of
// <d, q> follow the blocks.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "tpmg_device.cuh"
#include "tpmg_internal.h"

namespace tpmg {
namespace {

struct Quad {
    float a[4];
};

__device__ __forceinline__ Quad ld(const float *p)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return {{v.x, v.y, v.z, v.w}};
}

__device__ __forceinline__ void st(float *p, const Quad &q)
{
    *reinterpret_cast<float4 *>(p) = make_float4(q.a[0], q.a[1], q.a[2], q.a[3]);
}

template <bool BZ>
struct Loads {
    Quad z, zn, zs, tx, tn, ts, tz, h;
    Quad d[1], dn, ds;  // d_old (unset for BZ)
    float ze, zw, de, dw, tw;
};

template <bool BZ>
__global__ void __launch_bounds__(kBlock, 4)
k_dir_quad(LevelDev<float> L, const float *__restrict__ z, const float *__restrict__ d_even,
           const CgScalars *__restrict__ sc, float *__restrict__ d_to, float *__restrict__ q,
           int kz, double *__restrict__ partial, const int *__restrict__ flag,
           const CgLoop *__restrict__ loop)
{
    if (flag && !*flag) return;
    const bool odd = loop && (loop->its & 1);
    const float *__restrict__ dold = loop && loop->its == 0 ? z : odd ? d_to : d_even;
    float *__restrict__ dnew = odd ? const_cast<float *>(d_even) : d_to;
    const int nlon = L.nlon, nlat = L.nlat, nz = L.nz, nq = nlon / 4;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    float acc = 0.f;
    if (t < nq * nlat) {
        const int j = t / nq, i = 4 * (t - j * nq);
        const bool hasN = j + 1 < nlat, hasS = j > 0;
        const int dE = i + 4 == nlon ? -i : 4, dW = i == 0 ? nlon - 1 : -1;
        const size_t plane = (size_t)nlon * nlat, col = (size_t)j * nlon + i;
        const int k0 = blockIdx.y * kz, k1 = min(nz, k0 + kz);
        const float beta = BZ ? 0.f : (float)sc->beta;
        const Quad zero = {{0.f, 0.f, 0.f, 0.f}};
        auto load = [&](Loads<BZ> &l, int k) {
            const size_t o = (size_t)k * plane + col;
            l.z = ld(z + o);
            l.zn = hasN ? ld(z + o + nlon) : zero;
            l.zs = hasS ? ld(z + o - nlon) : zero;
            l.ze = __ldg(z + o + dE);
            l.zw = __ldg(z + o + dW);
            if (!BZ) {
                l.d[0] = ld(dold + o);
                l.dn = hasN ? ld(dold + o + nlon) : zero;
                l.ds = hasS ? ld(dold + o - nlon) : zero;
                l.de = __ldg(dold + o + dE);
                l.dw = __ldg(dold + o + dW);
            }
            l.tx = ld(L.tx + o);
            l.tw = __ldg(L.tx + o + dW);
            l.tn = hasN ? ld(L.ty + o) : zero;
            l.ts = hasS ? ld(L.ty + o - nlon) : zero;
            l.tz = ld(L.tz + o);
            l.h = ld(L.h + o);
        };
        auto dv = [&](float zv, float dvv) { return BZ ? zv : fmaf(beta, dvv, zv); };
        Quad xdn = zero, tdn = zero;
        if (k0 > 0) {
            const size_t o = (size_t)(k0 - 1) * plane + col;
            const Quad zb = ld(z + o), db = BZ ? zero : ld(dold + o);
            tdn = ld(L.tz + o);
#pragma unroll
            for (int e = 0; e < 4; ++e) xdn.a[e] = dv(zb.a[e], db.a[e]);
        }
        auto step = [&](const Loads<BZ> &c, Loads<BZ> &n, int k) {
            load(n, min(k + 1, nz - 1));  // in flight while layer k is combined
            Quad x, v;
#pragma unroll
            for (int e = 0; e < 4; ++e) x.a[e] = dv(c.z.a[e], c.d[0].a[e]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float xc = x.a[e];
                const float xe = e < 3 ? x.a[e < 3 ? e + 1 : 3] : dv(c.ze, c.de);
                const float xw = e > 0 ? x.a[e > 0 ? e - 1 : 0] : dv(c.zw, c.dw);
                float s = c.h.a[e] * xc;
                s = fmaf(c.tx.a[e], xc - xe, s);
                s = fmaf(e > 0 ? c.tx.a[e > 0 ? e - 1 : 0] : c.tw, xc - xw, s);
                if (hasN) s = fmaf(c.tn.a[e], xc - dv(c.zn.a[e], c.dn.a[e]), s);
                if (hasS) s = fmaf(c.ts.a[e], xc - dv(c.zs.a[e], c.ds.a[e]), s);
                const float xup = k + 1 < nz ? dv(n.z.a[e], n.d[0].a[e]) : 0.f;
                s = fmaf(c.tz.a[e], xc - xup, s);
                s = fmaf(tdn.a[e], xc - xdn.a[e], s);
                v.a[e] = s;
                acc = fmaf(s, xc, acc);
            }
            const size_t o = (size_t)k * plane + col;
            st(dnew + o, x);
            st(q + o, v);
            xdn = x;
            tdn = c.tz;
        };
        Loads<BZ> a, b;
        if (BZ) a.d[0] = b.d[0] = a.dn = a.ds = b.dn = b.ds = zero;
        if (BZ) a.de = a.dw = b.de = b.dw = 0.f;
        load(a, k0);
        for (int k = k0; k < k1; k += 2) {
            step(a, b, k);
            if (k + 1 < k1) step(b, a, k + 1);
        }
    }
    block_store_at<0>((double)acc, partial, blockIdx.y * gridDim.x + blockIdx.x);
}

struct Shape {
    int gx, gy, kz;
};

// Blocks along the columns, and the layers split until there are two waves of
// four blocks per SM: of a fixed number of SMs, since a batch lays out its
// partial sums (dir_quad_blocks) before it asks for a device.
constexpr long long kFillBlocks = 8 * 152;

Shape shape_of(const LevelDev<float> &L)
{
    Shape s;
    s.gx = (int)(((long long)(L.nlon / 4) * L.nlat + kBlock - 1) / kBlock);
    s.kz = L.nz;
    while (s.kz > 8 && (long long)s.gx * ((L.nz + s.kz - 1) / s.kz) < kFillBlocks)
        s.kz = (s.kz + 1) / 2;
    s.gy = (L.nz + s.kz - 1) / s.kz;
    return s;
}

}  // namespace

int dir_quad_blocks(const LevelDev<float> &L, const float *z, const float *d_old,
                    const float *d_new, const float *q)
{
    if (L.nlon % 4) return -1;
    uintptr_t p = 0;
    for (const void *v : {(const void *)z, (const void *)d_old, (const void *)d_new,
                          (const void *)q, (const void *)L.tx, (const void *)L.ty,
                          (const void *)L.tz, (const void *)L.h})
        p |= (uintptr_t)v;
    const Shape s = shape_of(L);
    return p % 16 || (long long)s.gx * s.gy > kReduceSlots ? -1 : s.gx * s.gy;
}

int launch_dir_quad(const LevelDev<float> &L, const float *z, const float *d_old,
                    const CgScalars *sc, float *d_new, float *q, double *partial, cudaStream_t s,
                    const int *flag, const CgLoop *loop)
{
    const int blocks = dir_quad_blocks(L, z, d_old, d_new, q);
    if (blocks < 0) return -1;
    const Shape g = shape_of(L);
    if (d_old)
        k_dir_quad<false><<<dim3(g.gx, g.gy), kBlock, 0, s>>>(L, z, d_old, sc, d_new, q, g.kz,
                                                              partial, flag, loop);
    else
        k_dir_quad<true><<<dim3(g.gx, g.gy), kBlock, 0, s>>>(L, z, d_old, sc, d_new, q, g.kz,
                                                             partial, flag, loop);
    return blocks;
}

}  // namespace tpmg
