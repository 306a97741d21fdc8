// Cone-beam forward and transpose over detector columns (cone_cols.cuh).
//
// Because every row of a detector column takes the same in-plane path, the
// in-plane part of Joseph's sample (split, weights, addresses) is common to a
// whole column, and along z the rays of a column on one plane are equally
// spaced.  Both kernels put the 32 lanes of a warp along z.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cone_cols.cuh"
#include "f32x2.cuh"

namespace psps {
namespace {

constexpr int kThreads = 256;

// ------------------------------------------------------------------ packing

// Border cells of the copies (kPad cells on every side of b and c), P floats
// each: per plane, 2 kPad full lines along the fast axis and n segments of
// 2 kPad cells, n the extent of the slow one.  c_fast: cells ordered [b][c],
// else [c][b].
__global__ void cone_border_kernel(int P, int nx, int ny, int nz, int copies, bool c_fast, float *__restrict__ ox,
                                   float *__restrict__ oy, float *__restrict__ oz) {
    constexpr int W = 2 * kPad;
    for (int a = 0; a < copies; ++a) {
        const int na = a == 0 ? nx : (a == 1 ? ny : nz);
        const int nb = a == 0 ? ny : nx, nc = a == 2 ? ny : nz;
        const int ns = c_fast ? nb : nc, nf = c_fast ? nc : nb, nsp = ns + W, nfp = nf + W;
        float *o = a == 0 ? ox : (a == 1 ? oy : oz);
        const int per = W * nfp + ns * W;                 // border cells of one plane
        const int64_t n = (int64_t)na * per;
        for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
            const int i = (int)(k / per), r = (int)(k - (int64_t)i * per);
            int s, f;
            if (r < W * nfp) {
                s = r / nfp;
                f = r - s * nfp;
                if (s >= kPad) s += ns;
            } else {
                const int q = r - W * nfp;
                s = kPad + q / W;
                f = q % W;
                if (f >= kPad) f += nf;
            }
            float *d = o + (((int64_t)i * nsp + s) * nfp + f) * P;
            for (int m = 0; m < P; ++m) d[m] = 0.f;
        }
    }
}

// Interiors of the x- and y-driven copies: a CTA turns a 32 x 32 (x, z) tile
// of one y around through shared memory, so that both sides are coalesced
// (x is fastest in the volume, z in the copies).  One read of the volume for
// both copies.
template <int P>
__global__ void __launch_bounds__(kThreads)
    cone_pack_kernel(const float *__restrict__ x, int nm, int nx, int ny, int nz, typename CPack<P>::T *__restrict__ ox,
                     typename CPack<P>::T *__restrict__ oy) {
    __shared__ float t[P][32][33];
    const int x0 = blockIdx.x * 32, z0 = blockIdx.z * 32, y = blockIdx.y;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t npix = (int64_t)nx * ny * nz;
    for (int r = wid; r < 32; r += kThreads / 32) {
        const int z = z0 + r, ix = x0 + lane;
        const bool in = z < nz && ix < nx;
#pragma unroll
        for (int m = 0; m < P; ++m)
            t[m][r][lane] = in && m < nm ? __ldg(x + m * npix + ((int64_t)z * ny + y) * nx + ix) : 0.f;
    }
    __syncthreads();
    const int z = z0 + lane;
    if (z >= nz) return;
    const int64_t ncp = nz + 2 * kPad;
    for (int r = wid; r < 32; r += kThreads / 32) {
        const int ix = x0 + r;
        if (ix >= nx) break;
        float v[P];
#pragma unroll
        for (int m = 0; m < P; ++m) v[m] = t[m][lane][r];
        typename CPack<P>::T o;
        if constexpr (P == 1) o = v[0];
        if constexpr (P == 2) o = make_float2(v[0], v[1]);
        if constexpr (P == 4) o = make_float4(v[0], v[1], v[2], v[3]);
        ox[((int64_t)ix * (ny + 2 * kPad) + y + kPad) * ncp + z + kPad] = o;
        oy[((int64_t)y * (nx + 2 * kPad) + ix + kPad) * ncp + z + kPad] = o;
    }
}

// Interiors of the copies ordered [c][b] (x fastest in the volume and in all but
// the x-driven copy); oz only with z-driven rays.
__global__ void cone_pack_rows_kernel(const float *__restrict__ x, int nm, int P, int nx, int ny, int nz,
                                      float *__restrict__ ox, float *__restrict__ oy, float *__restrict__ oz) {
    constexpr int W = 2 * kPad;
    const int64_t n = (int64_t)nx * ny * nz;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int ix = (int)(j % nx), iy = (int)((j / nx) % ny), iz = (int)(j / ((int64_t)nx * ny));
        float *dx = ox + (((int64_t)ix * (nz + W) + iz + kPad) * (ny + W) + iy + kPad) * P;
        float *dy = oy + (((int64_t)iy * (nz + W) + iz + kPad) * (nx + W) + ix + kPad) * P;
        float *dz = oz ? oz + (((int64_t)iz * (ny + W) + iy + kPad) * (nx + W) + ix + kPad) * P : nullptr;
        for (int m = 0; m < P; ++m) {
            const float v = m < nm ? x[m * n + j] : 0.f;
            dx[m] = v;
            dy[m] = v;
            if (dz) dz[m] = v;
        }
    }
}

// ------------------------------------------------------------------ forward

// One warp per detector column, lanes on neighbouring rows, R rows 32 apart
// per thread: the in-plane split and the addresses of the two volume lines it
// interpolates are the warp's, once per plane for 32 R rays, and a tap load
// reads neighbouring z of one line (rows are about one voxel apart), a few
// sectors, where lanes along the detector columns touched one line each.
// The taps of the next plane are loaded before those of this one are used
// (two register sets, the loop unrolled by two; 128 registers).  The samples
// of kSub planes are summed in FP32 and that partial is added to a
// Kahan-compensated total.  Results leave through shared memory so that each
// 8-column group writes whole 32-byte sectors.
// Bound by L1 latency and issue.  Two materials, 256^3 from 360 x 384 x 512
// rays: 12.6 ms (29.2 ms with one thread per ray along the detector rows,
// whose four taps touched 10.8 sectors per request against 6.2 here); 128^3
// from 180 x 192 x 256: 0.85 ms (1.80).  Tried: one register set (15.1 ms,
// long-scoreboard stalls), the plane's lines staged in shared memory by 16-byte
// asynchronous copies (22 ms: a third more instructions and a barrier per
// plane).
constexpr int kFCols = 8;    // detector columns (warps) per CTA
constexpr int kSub = 4;      // planes per compensated add

template <int NM, int R>
struct PlaneTaps {
    typename CPack<NM>::T t00[R], t01[R], t10[R], t11[R];
    float gc[R], gb;
};

template <int NM, int R>
__global__ void __launch_bounds__(32 * kFCols, 2)
    fwd_cols_kernel(mbir_geometry g, const float4 *__restrict__ col, const float2 *__restrict__ colw,
                    const typename CPack<NM>::T *__restrict__ ox, const typename CPack<NM>::T *__restrict__ oy, int nm,
                    int ncg, int64_t n_rays, float *__restrict__ l) {
    using T = typename CPack<NM>::T;
    constexpr int Rows = 32 * R;
    // sums as pairs: two rows of the one material, or two materials of a row
    constexpr int NP = NM == 1 ? R / 2 : R * NM / 2;
    static_assert(NM > 1 || R % 2 == 0, "rows pair up");
    __shared__ float out[NM][Rows][kFCols + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int v = blockIdx.x / ncg, u0 = (blockIdx.x - v * ncg) * kFCols, iu = u0 + wid, r0 = blockIdx.y * Rows;
    if (iu < g.n_u) {
        const float4 C = __ldg(col + (int64_t)v * g.n_u + iu);
        const float2 W = __ldg(colw + (int64_t)v * g.n_u + iu);
        int axis, lo, hi;
        decode_col(W, axis, lo, hi);
        const T *src = axis == 0 ? ox : oy;
        const int na = axis == 0 ? g.nx : g.ny, nb = axis == 0 ? g.ny : g.nx, nc = g.nz;
        const int nbp = nb + 2 * kPad, ncp = nc + 2 * kPad, cb = (nb >> 1) + kPad, cc = (nc >> 1) + kPad;
        const float ca = 0.5f * (na - 1), zo = cone_z_offset(nc), rc = 0.5f * (g.n_v - 1);
        float row[R];
        float klim = 0.f;   // largest k at which one of this thread's rays is still inside (-1, n_z)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int iv = r0 + lane + 32 * r;
            row[r] = (float)iv - rc;
            if (iv < g.n_v) klim = fmaxf(klim, __fdividef(0.5f * nc + 1.f, fmaxf(fabsf(row[r]), 1e-3f)));
        }
        // planes with k(t) = q0 + t dq below the warp's klim, one plane of margin
        klim = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(klim)));
        const float te = fminf(fmaxf((klim - C.z) / C.w + ca, -1.f), (float)na);
        if (C.w > 0.f)
            hi = min(hi, (int)ceilf(te) + 1);
        else
            lo = max(lo, (int)floorf(te) - 1);
        f32x2 acc[NP], comp[NP], part[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) acc[q] = comp[q] = part[q] = 0ull;
        const int64_t plane = (int64_t)nbp * ncp;
        auto fetch = [&](int i, PlaneTaps<NM, R> &p) {
            const float t = (float)i - ca;
            // indices clamped to the padded copy: a sample the clamp moves
            // lies outside the volume and reads border zeros, as it should
            const int ib = __vimin_s32_relu(joseph_split(fmaf(t, C.y, C.x), p.gb) + cb, nbp - 2);
            const float k = fmaf(t, C.w, C.z);
            const T *line = src + (i * plane + ib * ncp), *line1 = line + ncp;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int ic = __vimin_s32_relu(joseph_split(fmaf(row[r], k, zo), p.gc[r]) + cc, ncp - 2);
                p.t00[r] = __ldg(line + ic);
                p.t01[r] = __ldg(line + ic + 1);
                p.t10[r] = __ldg(line1 + ic);
                p.t11[r] = __ldg(line1 + ic + 1);
            }
        };
        auto use = [&](const PlaneTaps<NM, R> &p) {
            const f32x2 gb2 = pair2(p.gb, p.gb);
            auto sample = [&](f32x2 gc2, f32x2 a, f32x2 b, f32x2 c, f32x2 d, f32x2 &o) {
                const f32x2 e = fma2(gc2, sub2(b, a), a), f = fma2(gc2, sub2(d, c), c);
                o = add2(o, fma2(gb2, sub2(f, e), e));
            };
            if constexpr (NM == 1) {
#pragma unroll
                for (int r = 0; r < R; r += 2)
                    sample(pair2(p.gc[r], p.gc[r + 1]), pair2(p.t00[r], p.t00[r + 1]), pair2(p.t01[r], p.t01[r + 1]),
                           pair2(p.t10[r], p.t10[r + 1]), pair2(p.t11[r], p.t11[r + 1]), part[r / 2]);
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const f32x2 gc2 = pair2(p.gc[r], p.gc[r]);
                    sample(gc2, pair2(p.t00[r].x, p.t00[r].y), pair2(p.t01[r].x, p.t01[r].y),
                           pair2(p.t10[r].x, p.t10[r].y), pair2(p.t11[r].x, p.t11[r].y), part[r * NM / 2]);
                    if constexpr (NM == 4)
                        sample(gc2, pair2(p.t00[r].z, p.t00[r].w), pair2(p.t01[r].z, p.t01[r].w),
                               pair2(p.t10[r].z, p.t10[r].w), pair2(p.t11[r].z, p.t11[r].w), part[r * 2 + 1]);
                }
            }
        };
        auto flush = [&] {
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const f32x2 yk = sub2(part[q], comp[q]), tt = add2(acc[q], yk);
                comp[q] = sub2(sub2(tt, acc[q]), yk);
                acc[q] = tt;
                part[q] = 0ull;
            }
        };
        if (lo <= hi) {
            PlaneTaps<NM, R> p0, p1;
            fetch(lo, p0);
            int i = lo;
            for (; i < hi; i += 2) {
                fetch(i + 1, p1);
                use(p0);
                fetch(min(i + 2, hi), p0);
                use(p1);
                if ((i - lo) & (kSub - 2)) flush();
            }
            if (i == hi) use(p0);
            flush();
        }
        const float u = (float)((iu - 0.5 * (g.n_u - 1)) * g.du);
        float w[R];
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = cone_weight(g, W, u, row[r] * (float)g.dv);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            float a, b;
            unpair2(acc[q], a, b);
            if constexpr (NM == 1) {
                out[0][lane + 64 * q][wid] = a * w[2 * q];
                out[0][lane + 64 * q + 32][wid] = b * w[2 * q + 1];
            } else {
                constexpr int H = NM / 2;
                const int r = q / H, m = (q % H) * 2;
                out[m][lane + 32 * r][wid] = a * w[r];
                out[m + 1][lane + 32 * r][wid] = b * w[r];
            }
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < Rows * kFCols; q += 32 * kFCols) {
        const int rr = q / kFCols, cu = q % kFCols, iv = r0 + rr;
        if (iv >= g.n_v || u0 + cu >= g.n_u) continue;
        const int64_t ray = ((int64_t)v * g.n_v + iv) * g.n_u + u0 + cu;
#pragma unroll
        for (int m = 0; m < NM; ++m)
            if (m < nm) l[(int64_t)m * n_rays + ray] = out[m][rr][cu];
    }
}

// ------------------------------------------------------------------ transpose

// Weighted sinogram for the transpose, rows fastest:
// ws[(v n_u + iu) (n_v + 2 kRowPad) + kRowPad + iv][C], zero for the kRowPad
// rows on both sides, channels past nc zero.  32 x 32 (iu, iv) tiles through
// shared memory.  smax[c] (zeroed by the caller): max |ws| as float bits, NaN
// above every finite value.
template <int C>
__global__ void __launch_bounds__(kThreads)
    weigh_cols_kernel(mbir_geometry g, const float2 *__restrict__ colw, const float *__restrict__ sino, int nc,
                      int64_t n_rays, int ntu, int ntv, float *__restrict__ ws, unsigned *__restrict__ smax) {
    __shared__ float t[C][32][33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t n_tiles = (int64_t)g.n_views * ntu * ntv;
    const int stride = g.n_v + 2 * kRowPad;
    unsigned mx[C];
#pragma unroll
    for (int c = 0; c < C; ++c) mx[c] = 0u;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int v = (int)(tile / (ntu * ntv)), q = (int)(tile - (int64_t)v * ntu * ntv);
        const int u0 = (q % ntu) * 32, v0 = (q / ntu) * 32 - kRowPad;   // tiles cover the padded rows
        const int iu = u0 + lane;
        const float2 W = iu < g.n_u ? __ldg(colw + (int64_t)v * g.n_u + iu) : make_float2(0.f, 0.f);
        const float u = (float)((iu - 0.5 * (g.n_u - 1)) * g.du);
        for (int r = wid; r < 32; r += kThreads / 32) {
            const int iv = v0 + r;
            const bool in = iu < g.n_u && iv >= 0 && iv < g.n_v;
            const float w = cone_weight(g, W, u, ((float)iv - 0.5f * (g.n_v - 1)) * (float)g.dv);
            const int64_t ray = ((int64_t)v * g.n_v + iv) * g.n_u + iu;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const float val = in && c < nc ? w * __ldg(sino + c * n_rays + ray) : 0.f;
                const float a = fabsf(val);
                const unsigned bits = a != a ? 0x7fc00000u : __float_as_uint(a);
                mx[c] = bits > mx[c] ? bits : mx[c];
                t[c][r][lane] = val;
            }
        }
        __syncthreads();
        const int iv = v0 + lane;
        for (int r = wid; r < 32; r += kThreads / 32) {
            if (u0 + r >= g.n_u || iv >= g.n_v + kRowPad) continue;
            float *d = ws + (((int64_t)v * g.n_u + u0 + r) * stride + kRowPad + iv) * C;
            if constexpr (C == 4)
                *reinterpret_cast<float4 *>(d) = make_float4(t[0][lane][r], t[1][lane][r], t[2][lane][r], t[3][lane][r]);
            else
                *reinterpret_cast<float2 *>(d) = make_float2(t[0][lane][r], t[1][lane][r]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const unsigned m = __reduce_max_sync(0xffffffffu, mx[c]);
        if (lane == 0 && m) atomicMax(smax + c, m);
    }
}

// Detector columns whose rays, driven along A, can reach voxels of the patch
// [x0, x0 + kP) x [y0, y0 + kP) (clipped to the volume): the patch's footprint
// (exact on the driving axis, one voxel of margin on the interpolated one)
// projected onto the detector, widened by 1e-3 of a cell for rounding.
constexpr int kP = 4;   // patch side

template <int A>
__device__ __forceinline__ int2 patch_columns(const mbir_geometry &g, float4 V, int x0, int y0) {
    const float dx = (float)g.dx, dy = (float)g.dy, sdd = (float)g.sdd;
    const int x1 = min(x0 + kP, g.nx) - 1 + A, y1 = min(y0 + kP, g.ny) - A;
    const float xa = ((float)(x0 - A) - 0.5f * (g.nx - 1)) * dx, xb = ((float)x1 - 0.5f * (g.nx - 1)) * dx;
    const float ya = ((float)(y0 - 1 + A) - 0.5f * (g.ny - 1)) * dy, yb = ((float)y1 - 0.5f * (g.ny - 1)) * dy;
    float umin = 3.0e38f, umax = -3.0e38f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float qx = ((k & 1) ? xb : xa) - V.x, qy = ((k >> 1) ? yb : ya) - V.y;
        const float u = (-qx * V.w + qy * V.z) * (sdd / -(qx * V.z + qy * V.w));
        umin = fminf(umin, u);
        umax = fmaxf(umax, u);
    }
    const float inv = (float)(1.0 / g.du), cu = 0.5f * (g.n_u - 1);
    return make_int2(max((int)ceilf(fmaxf(umin * inv + cu - 1.0e-3f, -1.0f)), 0),
                     min((int)floorf(fminf(umax * inv + cu + 1.0e-3f, (float)g.n_u)), g.n_u - 1));
}

// Voxel-driven transpose.  A thread owns a kP x kP patch of (x, y) at one z,
// its warp 32 consecutive z.  For a view and a detector column whose rays
// cross the patch, the thread loads the NR rows around its z (their values do
// not change along the column), and on each of the patch's kP driving planes
// forms
//   T[c] = sum_rows max(0, 1 - |z_row - z|) ws[row][c],
// the transposed interpolation along z, which goes with the column's in-plane
// weights to the voxels of the plane that the column runs between.  What is
// common to the warp -- the in-plane weights of the plane's kP voxels and the
// row spacing k, per (column, plane) -- is worked out with one lane per pair,
// eight columns at a time, and read back from shared memory as broadcasts;
// all kP weights are applied (most are zero), which costs less than branching
// to the two that are not.  The accumulators stay in registers and there are
// no atomics.  FP32 sums run over kGroup views and are then added to the
// thread's totals in shared memory, with the rounding of every such add kept
// and put back in the next (a compensation of 8 significant bits below the
// total's 24, so the totals still leave room for 16 warps per SM; 32-bit
// compensations leave room for 12 and take 28.2 ms where this takes 23.9).
// The image is written once, or, when the views are split over blockIdx.y so
// that a small volume fills the GPU, as one partial image per split that
// cols_reduce_kernel adds in a fixed order.
// Either way the result does not depend on the order in which the CTAs run.
// Why so exact: the cross-material Fourier and wavelet preconditioners
// difference two materials' gradients after a spatial filter.  Relative error
// of the filtered gradient near convergence, 128^3, 180 / 720 views: plain
// totals of 32-view sums 7.7e-6 / 16.6e-6, this 4.8e-6 / 10.2e-6 (kGroup = 16:
// 5.5e-6 / 11.0e-6), the tile scatter with low words 5.8e-6 / 11.5e-6.
// Channel pairs use the packed operations.
// Bound by the shared-memory / L1 pipe (64 % busy, mostly the row loads: 16
// sectors each) and the latency its 16 warps per SM leave exposed.  Four
// channels, 256^3 from 360 x 384 x 512 rays: 23.9 ms with the weighting pass
// (77.7 ms for the ray-driven tile scatter); 128^3 from 180 x 192 x 256: 1.77 ms
// (5.3).  Two channels: 16.2 and 1.17 ms.  The compensated totals are 6 % of
// the four-channel times.  With plain totals, a branch to the two voxels with
// nonzero weight instead of all four weights took 29 ms (22.4) at 256^3, CTAs of 8
// and 16 warps, planes tested in pairs and an L1 prefetch of the next view's
// rows were no faster.
constexpr int kBX = 2, kBY = 2, kBWarps = kBX * kBY;   // warps per CTA: kBX x kBY patches of the same 32 z

struct ColDesc {                 // of (column q / kP, plane q % kP) of the current eight columns
    float4 wa[32], wb[32];       // in-plane weights of voxels 0..3, each twice
    float2 k[32];                // row spacing on the plane (0: no voxel reached), 1 / spacing on the middle plane
};

// One column: NR rows on the patch's kP planes, row `skip` of the window that
// starts at the row nearest (z's row) - first being the first of them.  The
// window's start is rounded once per z and column, whatever the pass: starts
// rounded pass by pass need not be whole passes apart (FP32 values of
// different binades), which lost or doubled a row at the seam.  src: row 0 of
// the column; wide: rows of the window before the last pass (0: one pass).
template <int A, int C, int NR, bool MULTI>
__device__ __forceinline__ void cols_column(const float *__restrict__ src, const float2 *dk, const float4 *da,
                                            const float4 *db, float mz, float rc, float first, int skip, int wide,
                                            int n_v, f32x2 (&acc)[kP][kP][C / 2]) {
    float fr = fmaf(-mz, dk[0].y, rc - first);
    fr = fminf(fmaxf(fr, (float)-(NR + wide)), (float)n_v);
    const float rn = fr + kSplitMagic;
    int r0 = __float_as_int(rn) - __float_as_int(kSplitMagic);
    float w0 = (rn - kSplitMagic) - rc;
    if constexpr (MULTI) {
        r0 = min(max(r0 + skip, -NR), n_v);   // a pass wholly outside reads zero rows
        w0 = (float)r0 - rc;
    }
    src += r0 * C;
    f32x2 s[NR][C / 2];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if constexpr (C == 4) {
            const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2 *>(src) + r);
            s[r][0] = q.x, s[r][1] = q.y;
        } else {
            s[r][0] = __ldg(reinterpret_cast<const f32x2 *>(src) + r);
        }
    }
    // planes tested together (a uniform branch when no voxel is reached): one
    // by one with four channels; with two, testing costs more than it saves
    constexpr int kTest = C == 4 ? 1 : kP;
#pragma unroll
    for (int pp = 0; pp < kP; pp += kTest) {
        float k[kTest], any = 0.f;
#pragma unroll
        for (int e = 0; e < kTest; ++e) k[e] = dk[pp + e].x, any = fmaxf(any, k[e]);
        if (any == 0.f) continue;
#pragma unroll
        for (int e = 0; e < kTest; ++e) {
            const int p = pp + e;
            f32x2 T[C / 2];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const float w = __saturatef(1.f - fabsf(fmaf(w0 + (float)r, k[e], mz)));
                const f32x2 w2 = pair2(w, w);
#pragma unroll
                for (int h = 0; h < C / 2; ++h) T[h] = fma2(w2, s[r][h], r == 0 ? 0ull : T[h]);
            }
            const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(da + p);
            const ulonglong2 wb = *reinterpret_cast<const ulonglong2 *>(db + p);
            const f32x2 wy[kP] = {wa.x, wa.y, wb.x, wb.y};
#pragma unroll
            for (int q = 0; q < kP; ++q)
#pragma unroll
                for (int h = 0; h < C / 2; ++h) {
                    f32x2 &o = A == 0 ? acc[p][q][h] : acc[q][p][h];
                    o = fma2(wy[q], T[h], o);
                }
        }
    }
}

template <int A, int C, int NR, bool MULTI>
__device__ __forceinline__ void cols_gather(const mbir_geometry &g, const float4 *__restrict__ cv,
                                            const float2 *__restrict__ wv, const float *__restrict__ wsv, int ua, int ub,
                                            bool mixed, int x0, int y0, float mz, float zmax, float first, int skip,
                                            int wide, ColDesc &desc, f32x2 (&acc)[kP][kP][C / 2]) {
    static_assert(kP == 4, "a lane per (column, plane) pair of eight columns, four weights per descriptor");
    const int na = A == 0 ? g.nx : g.ny, nb = A == 0 ? g.ny : g.nx;
    const int a0 = A == 0 ? x0 : y0, b0 = (A == 0 ? y0 : x0) - (nb >> 1);
    const float t0 = (float)a0 - 0.5f * (na - 1);
    const int n_v = g.n_v, stride = n_v + 2 * kRowPad, lane = threadIdx.x & 31;
    const float rc = 0.5f * (n_v - 1);
    for (int ug = ua; ug <= ub; ug += 8) {
        unsigned few = 0u;   // pairs whose rows all lie among three
        __syncwarp();        // the previous descriptors' readers are done
        {
            const int u = ug + lane / kP;
            const float t = t0 + (float)(lane % kP);
            float wy[kP] = {0.f, 0.f, 0.f, 0.f}, k = 0.f, inv = 0.f;
            if (u <= ub && !(mixed && (__float_as_int(__ldg(&wv[u].y)) & 3) != A)) {
                const float4 K = __ldg(cv + u);
                float gb;
                const int j = joseph_split(fmaf(t, K.y, K.x), gb) - b0;   // lower voxel, relative to the patch
#pragma unroll
                for (int q = 0; q < kP; ++q) wy[q] = q == j ? 1.f - gb : (q == j + 1 ? gb : 0.f);
                const float kp = fmaf(t, K.w, K.z);
                if (j >= -1 && j < kP) k = kp;
                inv = __fdividef(1.f, fmaf(t0 + 0.5f * (kP - 1), K.w, K.z));
                // a row within one voxel of z lies within 1 / kp of z's row on this
                // plane, which is zmax |1 / kp - inv| at most from the middle plane's;
                // three rows centred to half a row reach 3 / 2 (less 0.01 for rounding)
                const float ip = __fdividef(1.f, kp);
                few = fmaf(zmax, fabsf(ip - inv), ip) <= 1.49f;
            }
            few = __ballot_sync(0xffffffffu, few);
            desc.wa[lane] = make_float4(wy[0], wy[0], wy[1], wy[1]);
            desc.wb[lane] = make_float4(wy[2], wy[2], wy[3], wy[3]);
            desc.k[lane] = make_float2(k, inv);
        }
        __syncwarp();
        const int nu = min(8, ub - ug + 1);
        for (int c = 0; c < nu; ++c) {
            const float *src = wsv + ((int64_t)(ug + c) * stride + kRowPad) * C;
            if (NR == 4 && (few >> (c * kP) & 15u) == 15u)
                cols_column<A, C, 3, false>(src, &desc.k[c * kP], &desc.wa[c * kP], &desc.wb[c * kP], mz, rc, 1.f, 0, 0, n_v,
                                            acc);
            else
                cols_column<A, C, NR, MULTI>(src, &desc.k[c * kP], &desc.wa[c * kP], &desc.wb[c * kP], mz, rc, first, skip,
                                             wide, n_v, acc);
        }
    }
}

constexpr int kGroup = 8;   // views per compensated add
static_assert(32 % kGroup == 0, "groups end with the views that a warp's lanes look up together");

// Compensations of a pair of totals, each rounded to its upper 16 bits.
__device__ __forceinline__ f32x2 unpack_low(unsigned v) {
    return pair2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}
__device__ __forceinline__ unsigned pack_low(f32x2 v) {
    float a, b;
    unpair2(v, a, b);
    unsigned d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

// MULTI: the rows that reach one z exceed NR, so several passes of NR.
template <int C, int NR, bool MULTI>
__global__ void __launch_bounds__(32 * kBWarps, C == 4 ? 4 : 5)
    back_cols_kernel(mbir_geometry g, const float4 *__restrict__ vt, const int *__restrict__ view_cols,
                     const float4 *__restrict__ col, const float2 *__restrict__ colw, const float *__restrict__ ws,
                     const unsigned *__restrict__ smax, int nrows, int vchunk, int nc, float *__restrict__ x,
                     int64_t part_stride, int accumulate) {
    constexpr int N = kP * kP * C;
    extern __shared__ float4 back_smem[];
    ColDesc *descs = reinterpret_cast<ColDesc *>(back_smem);
    f32x2(*tot)[32 * kBWarps] = reinterpret_cast<f32x2(*)[32 * kBWarps]>(descs + kBWarps);
    unsigned(*low)[32 * kBWarps] = reinterpret_cast<unsigned(*)[32 * kBWarps]>(tot + N / 2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // CTA (xt, yt, zt), x fastest
    const int nxt = (g.nx + kBX * kP - 1) / (kBX * kP), nyt = (g.ny + kBY * kP - 1) / (kBY * kP);
    const int xt = blockIdx.x % nxt, yt = (blockIdx.x / nxt) % nyt, zt = blockIdx.x / (nxt * nyt);
    const int x0 = (xt * kBX + wid % kBX) * kP, y0 = (yt * kBY + wid / kBX) * kP, z = zt * 32 + lane;
    if (x0 >= g.nx || y0 >= g.ny) return;
    ColDesc &desc = descs[wid];
    // height of the middle of the volume relative to this voxel's centre
    const float mz = 0.5f * (g.nz - 1) - (float)z;
    const float zmax = fmaxf(fabsf(0.5f * (g.nz - 1) - (float)(zt * 32)), fabsf(0.5f * (g.nz - 1) - (float)(zt * 32 + 31)));
    const int vbeg = blockIdx.y * vchunk, vend = min(vbeg + vchunk, g.n_views);
    const int64_t vstride = (int64_t)g.n_u * (g.n_v + 2 * kRowPad) * C;
#pragma unroll
    for (int q = 0; q < N / 2; ++q) tot[q][threadIdx.x] = 0ull, low[q][threadIdx.x] = 0u;
    f32x2 acc[kP][kP][C / 2];
#pragma unroll
    for (int a = 0; a < kP; ++a)
#pragma unroll
        for (int b = 0; b < kP; ++b)
#pragma unroll
            for (int c = 0; c < C / 2; ++c) acc[a][b][c] = 0ull;
    for (int vb = vbeg; vb < vend; vb += 32) {
        // lane q: the patch's columns in view vb + q, per driving axis
        int axes = 0;
        int2 ux = make_int2(0, -1), uy = make_int2(0, -1);
        if (vb + lane < vend) {
            axes = __ldg(view_cols + vb + lane);
            const float4 V = __ldg(vt + vb + lane);
            if (axes & 1) ux = patch_columns<0>(g, V, x0, y0);
            if (axes & 2) uy = patch_columns<1>(g, V, x0, y0);
        }
        const int nv = min(32, vend - vb);
        for (int q = 0; q < nv; ++q) {
            const int ax = __shfl_sync(0xffffffffu, axes, q);
            const int xa = __shfl_sync(0xffffffffu, ux.x, q), xb = __shfl_sync(0xffffffffu, ux.y, q);
            const int ya = __shfl_sync(0xffffffffu, uy.x, q), yb = __shfl_sync(0xffffffffu, uy.y, q);
            const int64_t cv = (int64_t)(vb + q) * g.n_u;
            const float *wsv = ws + (int64_t)(vb + q) * vstride;
            for (int r = 0; r < (MULTI ? nrows : 1); r += NR) {
                const float first = 0.5f * ((MULTI ? nrows : NR) - 1);
                const int wide = MULTI ? nrows - NR : 0;
                if (ax & 1)
                    cols_gather<0, C, NR, MULTI>(g, col + cv, colw + cv, wsv, xa, xb, ax == 3, x0, y0, mz, zmax, first, r,
                                                 wide, desc, acc);
                if (ax & 2)
                    cols_gather<1, C, NR, MULTI>(g, col + cv, colw + cv, wsv, ya, yb, ax == 3, x0, y0, mz, zmax, first, r,
                                                 wide, desc, acc);
            }
            if ((q + 1) % kGroup && q + 1 < nv) continue;
#pragma unroll
            for (int a = 0; a < kP; ++a)
#pragma unroll
                for (int b = 0; b < kP; ++b)
#pragma unroll
                    for (int h = 0; h < C / 2; ++h) {
                        const int k = (a * kP + b) * (C / 2) + h;
                        const f32x2 t0 = tot[k][threadIdx.x];
                        const f32x2 yk = sub2(acc[a][b][h], unpack_low(low[k][threadIdx.x])), t1 = add2(t0, yk);
                        low[k][threadIdx.x] = pack_low(sub2(sub2(t1, t0), yk));
                        tot[k][threadIdx.x] = t1;
                        acc[a][b][h] = 0ull;
                    }
        }
    }
    if (z >= g.nz) return;
    const int64_t npix = (int64_t)g.nx * g.ny * g.nz;
    for (int c = 0; c < nc; ++c) {
        const bool bad = !(__uint_as_float(__ldg(smax + c)) <= 3.0e38f);   // a NaN or infinity poisons its channel
        for (int b = 0; b < kP && y0 + b < g.ny; ++b)
            for (int a = 0; a < kP && x0 + a < g.nx; ++a) {
                float t[2];
                unpair2(tot[((a * kP + b) * C + c) / 2][threadIdx.x], t[0], t[1]);
                const float v = bad ? __int_as_float(0x7fc00000) : (c & 1 ? t[1] : t[0]);
                const int64_t o = (int64_t)c * npix + ((int64_t)z * g.ny + y0 + b) * g.nx + x0 + a;
                if (part_stride)
                    x[blockIdx.y * part_stride + o] = v;
                else
                    x[o] = accumulate ? x[o] + v : v;
            }
    }
}

// x (+)= the sum of ns partial images, in order.
__global__ void __launch_bounds__(kThreads)
    cols_reduce_kernel(const float *__restrict__ part, int ns, int64_t stride, int64_t n, float *__restrict__ x,
                       int accumulate) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.f, comp = 0.f;
        for (int k = 0; k < ns; ++k) {
            const float yk = __fsub_rn(__ldg(part + k * stride + i), comp);
            const float t = __fadd_rn(s, yk);
            comp = __fsub_rn(__fsub_rn(t, s), yk);
            s = t;
        }
        x[i] = accumulate ? x[i] + s : s;
    }
}

}  // namespace

mbir_status cone_pack_rows(mbir_plan *p, const float *x, int nm, int P, bool z_too, cudaStream_t s) {
    const mbir_geometry &g = p->g;
    float *ox = p->xcol.p, *oy = p->xrow.p, *oz = z_too ? p->xcol3.p : nullptr;
    cone_border_kernel<<<608, kThreads, 0, s>>>(P, g.nx, g.ny, g.nz, z_too ? 3 : 2, false, ox, oy, oz);
    PSPS_LAUNCH_CHECK();
    const int64_t b = cdiv(p->n_pix, kThreads);
    cone_pack_rows_kernel<<<(unsigned)std::min<int64_t>(b, 65535 * 8), kThreads, 0, s>>>(x, nm, P, g.nx, g.ny, g.nz, ox, oy,
                                                                                          oz);
    PSPS_LAUNCH_CHECK();
    return MBIR_OK;
}

// The copies ordered [b][c] that the columns read.
static mbir_status cone_pack(mbir_plan *p, const float *x, int nm, int P, cudaStream_t s) {
    const mbir_geometry &g = p->g;
    float *ox = p->xcol.p, *oy = p->xrow.p;
    cone_border_kernel<<<608, kThreads, 0, s>>>(P, g.nx, g.ny, g.nz, 2, true, ox, oy, nullptr);
    PSPS_LAUNCH_CHECK();
    const dim3 grd((unsigned)cdiv(g.nx, 32), (unsigned)g.ny, (unsigned)cdiv(g.nz, 32));
    if (P == 1)
        cone_pack_kernel<1><<<grd, kThreads, 0, s>>>(x, nm, g.nx, g.ny, g.nz, ox, oy);
    else if (P == 2)
        cone_pack_kernel<2><<<grd, kThreads, 0, s>>>(x, nm, g.nx, g.ny, g.nz, (float2 *)ox, (float2 *)oy);
    else
        cone_pack_kernel<4><<<grd, kThreads, 0, s>>>(x, nm, g.nx, g.ny, g.nz, (float4 *)ox, (float4 *)oy);
    PSPS_LAUNCH_CHECK();
    return MBIR_OK;
}

mbir_status cone_cols_setup(mbir_plan *p) {
    const mbir_geometry &g = p->g;
    p->cols = false;
    p->col_rows = 0;
    // z-driven rays exist only where |w| > max(|d_x|, |d_y|) >= sdd / sqrt 2
    p->cols = 0.5 * (g.n_v - 1) * g.dv < 0.999 * g.sdd / std::sqrt(2.0);
    if (!p->cols) return MBIR_OK;
    // Rows that can reach one z on the kP planes of a patch: on one plane the
    // rows are k = dv D / (sdd dz) voxels apart, D >= D_min = sid - R the depth
    // from the source, so those within one voxel lie within 1 / k of the
    // z's own row position; moving one plane changes D by at most
    // sqrt2 h (h the plane spacing), which moves that position, at most
    // (nz / 2 + 1) / k, by the fraction sqrt2 h / D_min; the patch's planes are
    // (kP - 1) / 2 from the middle one.  NR rows centred to half a row reach
    // NR / 2.
    // (R holds a patch's overhang beyond the volume.)
    const double R = std::hypot((0.5 * g.nx + kP) * g.dx, (0.5 * g.ny + kP) * g.dy), D = g.sid - R;
    if (!(D > 1e-3 * g.sid)) return MBIR_OK;
    const double k = g.dv * D / (g.sdd * g.dz);
    const double drift = (0.5 * g.nz + 1.0) * std::sqrt(2.0) * std::max(g.dx, g.dy) / D * 0.5 * (kP - 1);
    const double need = 2.0 * (1.0 + drift) / k + 0.02;
    if (g.n_v >= (1 << 20)) return MBIR_OK;   // the row search's FP32 indices
    // Its lanes run along z and every 32 layers cost the same, the tile scatter
    // costs in proportion to the rows, above a floor per view that small
    // images do not reach.  Two channels, us by tile / columns, as many rows as
    // layers: 512 x 512 from 180 views 8 rows 2910 / 2850, 12 rows 3890 / 2860;
    // 256 x 256 from 360 views 4 rows 1360 / 1850, 8 rows 1980 / 2020, 12 rows
    // 2660 / 2030; 128 x 128 from 180 views 4 rows 325 / 284, 8 rows 428 / 282;
    // four channels 256 x 256 8 rows 2450 / 2940, 12 rows 3350 / 2980, 128 x 128
    // 4 rows 362 / 393, 8 rows 501 / 401; 64 x 64 from 90 views 4 rows 186 / 82.
    const int64_t h = std::min<int64_t>(g.n_v / cdiv(g.nz, 32), g.nz);
    if (h < 4 || (h < 12 && (int64_t)g.nx * g.ny * 12 > (h + 4) * 128 * 128)) return MBIR_OK;
    if (need > 48.0) return MBIR_OK;
    p->col_rows = need <= 4.0 ? std::max(2, (int)std::ceil(need)) : 6 * (int)std::ceil(need / 6.0);
    // View splits: enough warps for about three waves of 16 per SM, at least
    // four views each, partial images of at most 256 MB.
    const int64_t warps = cdiv(g.nx, kP) * cdiv(g.ny, kP) * cdiv(g.nz, 32);
    const int64_t want = cdiv((int64_t)152 * 16 * 3, warps);
    const int64_t cap = std::max<int64_t>(1, ((int64_t)1 << 26) / (4 * p->n_pix));
    int64_t ns = std::min(std::min(want, cap), std::max<int64_t>(1, g.n_views / 4));
    p->col_vchunk = (int)cdiv(g.n_views, ns);
    p->col_splits = (int)cdiv(g.n_views, p->col_vchunk);
    return p->col_splits > 1 ? p->col_part.alloc((size_t)p->col_splits * 4 * p->n_pix) : MBIR_OK;
}

// A warp per detector column costs the same whatever the number of its rows
// that meet the volume, a thread per ray in proportion to it.  256 x 256 voxels
// from 360 x 512 columns, us per ray / columns, for as many rows (32 and 64
// per warp) as layers: one material 24 rows 1500 / 1940, 32 rows 1970 / 1940,
// 64 rows 3850 / 1950; two 12 rows 1090 / 1450, 16 rows 1440 / 1450, 24 rows
// 2130 / 1460; four 16 rows 1910 / 1940, 24 rows 2840 / 1950.  The lines lie at
// the same row counts for 64 to 512 voxels across and 60 to 360 views.
bool cone_cols_forward(const mbir_geometry &g, int P) {
    const double hit = std::min((double)g.n_v, g.nz * g.dz * g.sdd / (g.sid * g.dv));   // rows that meet the volume
    return hit >= (P == 1 ? 32.0 : 17.0);
}

mbir_status project_cone_cols(mbir_plan *p, const float *x, float *l, int nm, cudaStream_t s) {
    const mbir_geometry &g = p->g;
    const int P = nm == 1 ? 1 : (nm == 2 ? 2 : 4);
    PSPS_TRY(cone_pack(p, x, nm, P, s));
    const int ncg = (int)cdiv(g.n_u, kFCols);
    auto run = [&](auto m, auto r) {
        constexpr int M = decltype(m)::value, R = decltype(r)::value;
        using T = typename CPack<M>::T;
        const dim3 grd((unsigned)((int64_t)ncg * g.n_views), (unsigned)cdiv(g.n_v, 32 * R));
        fwd_cols_kernel<M, R><<<grd, 32 * kFCols, 0, s>>>(g, p->col.p, p->colw.p, reinterpret_cast<const T *>(p->xcol.p),
                                                          reinterpret_cast<const T *>(p->xrow.p), nm, ncg, p->n_rays, l);
    };
    // of two row counts the one whose last chunk wastes less (ties: more rows)
    auto pick = [&](auto m, auto r0, auto r1) {
        const int a = 32 * decltype(r0)::value, b = 32 * decltype(r1)::value;
        if (cdiv(g.n_v, a) * a <= cdiv(g.n_v, b) * b)
            run(m, r0);
        else
            run(m, r1);
    };
    // few rows: one chunk of 32 or 64, whose warps hold fewer idle rows
    using std::integral_constant;
    if (P == 1) {
        if (g.n_v <= 64)
            run(integral_constant<int, 1>{}, integral_constant<int, 2>{});
        else
            pick(integral_constant<int, 1>{}, integral_constant<int, 6>{}, integral_constant<int, 4>{});
    } else if (P == 2) {
        if (g.n_v <= 32)
            run(integral_constant<int, 2>{}, integral_constant<int, 1>{});
        else if (g.n_v <= 64)
            run(integral_constant<int, 2>{}, integral_constant<int, 2>{});
        else
            pick(integral_constant<int, 2>{}, integral_constant<int, 4>{}, integral_constant<int, 3>{});
    } else {
        pick(integral_constant<int, 4>{}, integral_constant<int, 2>{}, integral_constant<int, 1>{});
    }
    PSPS_LAUNCH_CHECK();
    return MBIR_OK;
}

namespace {

template <int C>
mbir_status backproject_cols(mbir_plan *p, const float *sino, float *x, int nc, int accumulate, cudaStream_t s) {
    const mbir_geometry &g = p->g;
    const int ntu = (int)cdiv(g.n_u, 32), ntv = (int)cdiv(g.n_v + 2 * kRowPad, 32);
    const int64_t tiles = (int64_t)g.n_views * ntu * ntv;
    PSPS_CUDA(cudaMemsetAsync(p->wmax.p, 0, C * sizeof(unsigned), s));
    weigh_cols_kernel<C><<<(unsigned)std::min<int64_t>(tiles, 152 * 8), kThreads, 0, s>>>(
        g, p->colw.p, sino, nc, p->n_rays, ntu, ntv, p->wsino.p, p->wmax.p);
    PSPS_LAUNCH_CHECK();
    const int ns = p->col_splits;
    const dim3 grd((unsigned)(cdiv(g.nx, kBX * kP) * cdiv(g.ny, kBY * kP) * cdiv(g.nz, 32)), (unsigned)ns);
    float *dst = ns > 1 ? p->col_part.p : x;
    const int64_t stride = ns > 1 ? (int64_t)4 * p->n_pix : 0;
    auto run = [&](auto nr, auto multi) -> mbir_status {
        constexpr size_t smem = kBWarps * (sizeof(ColDesc) + (sizeof(f32x2) + sizeof(unsigned)) * (kP * kP * C / 2) * 32);
        constexpr auto kernel = back_cols_kernel<C, decltype(nr)::value, decltype(multi)::value>;
        PSPS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kernel<<<grd, 32 * kBWarps, smem, s>>>(g, p->view.p, p->view_cols.p, p->col.p, p->colw.p, p->wsino.p, p->wmax.p,
                                               p->col_rows, p->col_vchunk, nc, dst, stride, accumulate);
        PSPS_LAUNCH_CHECK();
        return MBIR_OK;
    };
    switch (p->col_rows) {
        case 2: PSPS_TRY(run(std::integral_constant<int, 2>{}, std::false_type{})); break;
        case 3: PSPS_TRY(run(std::integral_constant<int, 3>{}, std::false_type{})); break;
        case 4: PSPS_TRY(run(std::integral_constant<int, 4>{}, std::false_type{})); break;
        default: PSPS_TRY(run(std::integral_constant<int, 6>{}, std::true_type{})); break;   // passes of 6
    }
    if (ns > 1) {
        const int64_t n = (int64_t)nc * p->n_pix, b = cdiv(n, kThreads);
        cols_reduce_kernel<<<(unsigned)(b < 4096 ? b : 4096), kThreads, 0, s>>>(p->col_part.p, ns, stride, n, x,
                                                                               accumulate);
        PSPS_LAUNCH_CHECK();
    }
    return MBIR_OK;
}

}  // namespace

mbir_status backproject_cone_cols(mbir_plan *p, const float *sino, float *x, int nc, int accumulate, cudaStream_t s) {
    return nc > 2 ? backproject_cols<4>(p, sino, x, nc, accumulate, s)
                  : backproject_cols<2>(p, sino, x, nc, accumulate, s);
}

}  // namespace psps
