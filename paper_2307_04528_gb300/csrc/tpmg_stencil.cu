// FP64 stencils (operator apply, residual, and the refinement's scaled FP32
// residual) with a thread per 2 x 2 columns walking a range of layers.
//
// The FP64 kernels are bound by the FP64 pipe (two lanes per SM and clock),
// so what counts is FP64 operations per cell.  In flux form each face's
// difference x_c - x_nb is needed by both of its cells, with opposite signs;
// a thread forms the differences between its own four columns once, and
// carries each vertical difference to the layer above: 4 subtractions per
// cell instead of 6 (11 operations instead of 13, 12 instead of 14 with the
// fused inner product).  A difference is exact up to its sign, so every value
// is the one the column walk (stencil_column) gives, bit for bit; only the
// grouping of the partial sums follows the blocks.  All own-cell loads are
// 16-byte pairs, one layer ahead of the arithmetic.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "tpmg_device.cuh"
#include "tpmg_internal.h"

namespace tpmg {
namespace {

// The operator: mass h (or the horizontal diagonal, HSUM), each cell's own
// couplings e, n, u to its east, north and upper neighbour, and the couplings
// w, s, d back to it, read at the west, south and lower neighbour's index
// (the symmetric operator: w = e, s = n, d = u).
struct StencilView {
    int nlon, nlat, nz;
    const double *h, *e, *n, *u, *w, *s, *d;
};

struct Two {
    double a[2];
};

__device__ __forceinline__ Two ld2(const double *p)
{
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {{v.x, v.y}};
}

// The same of x or b, which the kernel before this one may have written
// (after_previous).
__device__ __forceinline__ Two ld2_of(const double *p)
{
    const double2 v = *reinterpret_cast<const double2 *>(p);
    return {{v.x, v.y}};
}

// One layer of a thread's 2 x 2 columns: [row][column].
template <bool SYM, bool RESID>
struct Layer {
    Two x[2], h[2], e[2], n[2], u[2], b[RESID ? 2 : 1];
    Two w[SYM ? 1 : 2], s0[1], sr[SYM ? 1 : 2], d[SYM ? 1 : 2];
    double xw[2], xe[2], ew[2];
    Two xn, xs;
};

// RESID: y = b - A x, else A x.  RED: block sums of y y (RESID) or x y.
// CAST: y receives the FP32 rounding of the value times scale (NARROW: the
// scaling after the rounding, stencil_column).  HSUM: V.h holds the mass plus
// the four horizontal couplings and the horizontal terms are taken in sum
// form, as stencil_column.
template <bool SYM, bool RESID, bool RED, bool CAST, bool NARROW, bool HSUM>
__global__ void __launch_bounds__(kBlock, 3)
k_stencil_quad(StencilView V, const double *b, const double *x, void *__restrict__ yout,
               double scale, int kz, double *__restrict__ partial, const int *flag)
{
    after_previous();
    if (flag && !*flag) return;
    const int nlon = V.nlon, nlat = V.nlat, nz = V.nz, half = nlon / 2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    double acc = 0.0;
    if (t < half * (nlat / 2)) {
        const int jp = t / half, i = 2 * (t - jp * half), j = 2 * jp;
        const size_t plane = (size_t)nlon * nlat;
        const bool hasN = j + 2 < nlat, hasS = j > 0;
        const int dE = i + 2 == nlon ? -i : 2, dW = i == 0 ? nlon - 1 : -1;
        const size_t col = (size_t)j * nlon + i;
        const int k0 = blockIdx.y * kz, k1 = min(nz, k0 + kz);
        const Two zero = {{0.0, 0.0}};
        using L = Layer<SYM, RESID>;
        auto load = [&](L &l, int k) {
            const size_t o = (size_t)k * plane + col;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const size_t c = o + (size_t)r * nlon;
                l.x[r] = ld2_of(x + c);
                l.xe[r] = x[c + dE];
                l.xw[r] = x[c + dW];
                l.e[r] = ld2(V.e + c);
                l.ew[r] = __ldg(V.w + c + dW);
                l.n[r] = ld2(V.n + c);
                l.u[r] = ld2(V.u + c);
                l.h[r] = ld2(V.h + c);
                if (!SYM) {
                    l.w[SYM ? 0 : r] = ld2(V.w + c);
                    l.sr[SYM ? 0 : r] = ld2(V.s + c);
                    l.d[SYM ? 0 : r] = ld2(V.d + c);
                }
                if (RESID) l.b[RESID ? r : 0] = ld2_of(b + c);
            }
            l.xn = hasN ? ld2_of(x + o + 2 * (size_t)nlon) : zero;
            l.xs = hasS ? ld2_of(x + o - nlon) : zero;
            l.s0[0] = hasS ? ld2(V.s + o - nlon) : zero;
        };
        L cur, nxt;
        load(cur, k0);
        Two dn[2] = {zero, zero}, tdn[2] = {zero, zero};  // x_below - x and its coupling
        // below the surface x and its coupling count as zero, as above the top
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) dn[r].a[q] = -cur.x[r].a[q];
        if (k0 > 0)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const size_t c = (size_t)(k0 - 1) * plane + col + (size_t)r * nlon;
                const Two xb = ld2_of(x + c);
                tdn[r] = ld2(V.d + c);
#pragma unroll
                for (int q = 0; q < 2; ++q) dn[r].a[q] = xb.a[q] - cur.x[r].a[q];
            }
        for (int k = k0; k < k1; ++k) {
            if (k + 1 < nz) load(nxt, k + 1);  // x of the layer above; the next layer
            Two v[2];
            double ew0[2], nd[2];
            if (!HSUM) {
#pragma unroll
                for (int r = 0; r < 2; ++r) ew0[r] = cur.x[r].a[0] - cur.x[r].a[1];
#pragma unroll
                for (int q = 0; q < 2; ++q) nd[q] = cur.x[0].a[q] - cur.x[1].a[q];
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const double xc = cur.x[r].a[q];
                    const double te = cur.e[r].a[q];
                    const double tw = q == 0 ? cur.ew[r]
                                             : (SYM ? cur.e[r].a[0] : cur.w[SYM ? 0 : r].a[0]);
                    const double tn = cur.n[r].a[q];
                    const double ts = r == 0 ? cur.s0[0].a[q]
                                             : (SYM ? cur.n[0].a[q] : cur.sr[0].a[q]);
                    double s = cur.h[r].a[q] * xc;
                    if (HSUM) {
                        s = fma(-te, q == 0 ? cur.x[r].a[1] : cur.xe[r], s);
                        s = fma(-tw, q == 0 ? cur.xw[r] : cur.x[r].a[0], s);
                        if (r == 0 || hasN) s = fma(-tn, r == 0 ? cur.x[1].a[q] : cur.xn.a[q], s);
                        if (r == 1 || hasS) s = fma(-ts, r == 0 ? cur.xs.a[q] : cur.x[0].a[q], s);
                    } else {
                        s = fma(te, q == 0 ? ew0[r] : xc - cur.xe[r], s);
                        s = fma(tw, q == 0 ? xc - cur.xw[r] : -ew0[r], s);
                        if (r == 0 || hasN) s = fma(tn, r == 0 ? nd[q] : xc - cur.xn.a[q], s);
                        if (r == 1 || hasS) s = fma(ts, r == 0 ? xc - cur.xs.a[q] : -nd[q], s);
                    }
                    // x above the top counts as zero, its coupling is zero: no
                    // branch, whose two sides would both issue
                    const double up = xc - (k + 1 < nz ? nxt.x[r].a[q] : 0.0);
                    s = fma(cur.u[r].a[q], up, s);
                    s = fma(tdn[r].a[q], -dn[r].a[q], s);
                    dn[r].a[q] = up;
                    tdn[r].a[q] = SYM ? cur.u[r].a[q] : cur.d[SYM ? 0 : r].a[q];
                    const double out = RESID ? cur.b[RESID ? r : 0].a[q] - s : s;
                    if (RED) acc = fma(out, RESID ? out : xc, acc);
                    v[r].a[q] = out;
                }
                const size_t c = (size_t)k * plane + col + (size_t)r * nlon;
                if (CAST) {
                    float2 f;
                    f.x = NARROW ? f64_to_f32_rn(v[r].a[0]) * (float)scale
                                 : f64_to_f32_rn(v[r].a[0] * scale);
                    f.y = NARROW ? f64_to_f32_rn(v[r].a[1]) * (float)scale
                                 : f64_to_f32_rn(v[r].a[1] * scale);
                    *reinterpret_cast<float2 *>(static_cast<float *>(yout) + c) = f;
                } else {
                    *reinterpret_cast<double2 *>(static_cast<double *>(yout) + c) =
                        make_double2(v[r].a[0], v[r].a[1]);
                }
            }
            cur = nxt;
        }
    }
    if (RED) block_store_at<0>(acc, partial, blockIdx.y * gridDim.x + blockIdx.x);
}

int g_stencil_sms = 152;

struct Shape {
    int gx, gy, kz;
};

// Blocks along the columns, and the layers split until there are four blocks
// for every SM (256 x 128 x 32: 64 column blocks alone would leave half of
// the GPU idle).
Shape shape_of(int nlon, int nlat, int nz)
{
    Shape s;
    const long long quads = (long long)(nlon / 2) * (nlat / 2);
    s.gx = (int)((quads + kBlock - 1) / kBlock);
    s.kz = nz;
    while (s.kz > 4 && (long long)s.gx * ((nz + s.kz - 1) / s.kz) < 4LL * g_stencil_sms)
        s.kz = (s.kz + 1) / 2;
    s.gy = (nz + s.kz - 1) / s.kz;
    return s;
}

bool quad_fits(const StencilView &V, std::initializer_list<const void *> ptrs, const Shape &s)
{
    if (V.nlon % 2 || V.nlat % 2 || (long long)s.gx * s.gy > kReduceSlots) return false;
    uintptr_t p = 0;
    for (const void *q : ptrs) p |= (uintptr_t)q;
    return p % 16 == 0;
}

template <bool SYM>
int launch_view(const StencilView &V, int mode, const double *b, const double *x, double *y,
                double *partial, cudaStream_t s, const int *flag)
{
    const Shape g = shape_of(V.nlon, V.nlat, V.nz);
    if (!quad_fits(V, {V.h, V.e, V.n, V.u, V.w, V.s, V.d, b, x, y}, g)) return -1;
    const dim3 grid(g.gx, g.gy);
    if (mode && partial)
        launch_after(k_stencil_quad<SYM, true, true, false, false, false>, grid, kBlock, 0, s, V, b,
                     x, y, 1.0, g.kz, partial, flag);
    else if (mode)
        launch_after(k_stencil_quad<SYM, true, false, false, false, false>, grid, kBlock, 0, s, V,
                     b, x, y, 1.0, g.kz, nullptr, flag);
    else if (partial)
        launch_after(k_stencil_quad<SYM, false, true, false, false, false>, grid, kBlock, 0, s, V,
                     b, x, y, 1.0, g.kz, partial, flag);
    else
        launch_after(k_stencil_quad<SYM, false, false, false, false, false>, grid, kBlock, 0, s, V,
                     b, x, y, 1.0, g.kz, nullptr, flag);
    return g.gx * g.gy;
}

StencilView sym(const LevelDev<double> &L)
{
    return {L.nlon, L.nlat, L.nz, L.h, L.tx, L.ty, L.tz, L.tx, L.ty, L.tz};
}

}  // namespace

void stencil_prepare(int sms)
{
    if (sms > 0) g_stencil_sms = sms;
}

int launch_stencil_quad(const LevelDev<double> &L, int mode, const double *b, const double *x,
                        double *y, double *partial, cudaStream_t s, const int *flag)
{
    return launch_view<true>(sym(L), mode, b, x, y, partial, s, flag);
}

int launch_ns_stencil_quad(const NsView<double> &V, int mode, const double *b, const double *x,
                           double *y, cudaStream_t s)
{
    return launch_view<false>({V.nlon, V.nlat, V.nz, V.h, V.e, V.n, V.u, V.w, V.s, V.d}, mode, b,
                              x, y, nullptr, s, nullptr);
}

int launch_residual_cast_quad(const LevelDev<double> &L, const double *b, const double *x,
                              float *r32, double inv_scale, bool narrow, double *partial,
                              cudaStream_t s)
{
    const StencilView V = sym(L);
    const Shape g = shape_of(V.nlon, V.nlat, V.nz);
    if (!quad_fits(V, {V.h, V.e, V.n, V.u, b, x, r32}, g)) return -1;
    const dim3 grid(g.gx, g.gy);
    if (narrow)
        launch_after(k_stencil_quad<true, true, true, true, true, true>, grid, kBlock, 0, s, V, b,
                     x, r32, inv_scale, g.kz, partial, nullptr);
    else
        launch_after(k_stencil_quad<true, true, true, true, false, true>, grid, kBlock, 0, s, V, b,
                     x, r32, inv_scale, g.kz, partial, nullptr);
    return g.gx * g.gy;
}

}  // namespace tpmg
