// Templated per-ray kernels of the spectral model (model.cu): the data term
// with SPS numerators and the fused line-search evaluation, plain and with
// rays coupled along detector rows.  Each material count is instantiated in
// its own translation unit (model_inst.cu compiled once per count and
// family), so the 128 kernel variants compile in parallel.
#pragma once
#include <cmath>

#include "f32x2.cuh"
#include "model.cuh"

namespace psps {
namespace {

constexpr int kMaxE = 256, kMaxC = 8;

__device__ __forceinline__ void load_spec(const SpecDev &sp, float *sh) {
    const int n = sp.ne * sp.nm + sp.nc * sp.ne + sp.nc;
    for (int i = threadIdx.x; i < n; i += blockDim.x) sh[i] = sp.qs[i];
    __syncthreads();
}

// Channel counts are compile-time upper bounds CM (1, 2, 4, 8); channels nc..CM
// have zero sensitivity, so the per-channel accumulators stay in registers.
// t = exp(-z) through the base-2 exponential: exp2f(-z log2 e), with
// log2 e = 1 / ln 2.  exp2f maps to the SFU's base-2 exponential (2 ulp);
// the product adds a relative error of about |z| 2^-24 to t.
__device__ __forceinline__ float transmission(float z) { return exp2f(z * -1.4426950408889634f); }

// The energy loops take two rays per thread, as the two halves of packed FP32
// pairs, which halves the issue slots of everything but the exponentials.
// Their table holds, per energy, every factor twice (one 16-byte shared-memory
// load brings two of them, for both rays): Q[E][m], then S[c][E].  The exponent
// -log2(e) z of 2 is one more product per energy.  Putting the factor into the
// table (error of a one-energy gradient 7.8e-8 instead of 4.0e-8) or into the
// line integrals (two materials: 3.30e-7 instead of 3.17e-7, since a rounded
// line integral errs alike at every energy) saves that, 3 % of a
// projection-domain iteration.
// Measured on 720 x 888 rays, 2 materials, 121 energies, 2 channels, against one
// ray per thread with exp2f's subnormal handling and every channel at every
// energy: numerators 117 -> 84 us, line-search evaluation 76 -> 57 us (ncu, cold);
// 3 materials, 4 channels: model stage 148 -> 89 us, line search 508 -> 322 us per
// iteration, halvings included; with blur and correlated noise the data-term
// gradient 175 -> 100 us.  The FP32 pipe and issue are half busy (54 % and 52 %
// for the evaluation); more rays (x 8) run at the same rate.
constexpr float kLog2e = 1.4426950408889634f;

// Exponents of 2 that give exp(-z).
__device__ __forceinline__ f32x2 neglog2e(f32x2 z) { return mul2(z, pair2(-kLog2e, -kLog2e)); }

template <int NM, int CM>
struct SpecTab {
    static constexpr int Stride = (NM + CM + 1) & ~1;   // pairs per energy
    const f32x2 *rec;
    const float *sig;                                   // sigma[c]
    int ne, nc;
    const SpecSegs *segs;                               // of the kernel's (grid-constant) parameter

    __host__ __device__ static size_t bytes(int ne, int nc) { return sizeof(f32x2) * Stride * ne + sizeof(float) * ((nc + 3) & ~3); }

    __device__ __forceinline__ void load(const SpecDev &sp, void *smem) {
        f32x2 *r = static_cast<f32x2 *>(smem);
        float *sg = reinterpret_cast<float *>(r + Stride * sp.ne);
        ne = sp.ne, nc = sp.nc, rec = r, sig = sg, segs = &sp.segs;
        const float *S = sp.qs + sp.ne * NM;
        for (int i = threadIdx.x; i < ne * Stride; i += blockDim.x) {
            const int e = i / Stride, k = i - e * Stride;
            float v = 0.f;
            if (k < NM) {
                v = sp.qs[e * NM + k];
            } else if (k - NM < nc) {
                v = S[(k - NM) * ne + e];
            }
            r[i] = pair2(v, v);
        }
        for (int c = threadIdx.x; c < nc; c += blockDim.x) sg[c] = S[nc * ne + c];
        __syncthreads();
    }
    __device__ __forceinline__ void get(int e, f32x2 (&q)[NM], f32x2 (&s)[CM]) const {
        const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(rec + e * Stride);
        f32x2 v[Stride];
#pragma unroll
        for (int k = 0; k < Stride / 2; ++k) {
            const ulonglong2 w = p[k];
            v[2 * k] = w.x, v[2 * k + 1] = w.y;
        }
#pragma unroll
        for (int m = 0; m < NM; ++m) q[m] = v[m];
#pragma unroll
        for (int c = 0; c < CM; ++c) s[c] = v[NM + c];
    }
    // The factors q and the one sensitivity of channel c.
    __device__ __forceinline__ void get(int e, int c, f32x2 (&q)[NM], f32x2 &s) const {
        const f32x2 *p = rec + e * Stride;
#pragma unroll
        for (int m = 0; m < NM; ++m) q[m] = p[m];
        s = p[NM + c];
    }
};

template <int N>
__device__ __forceinline__ f32x2 dot2(const f32x2 (&a)[N], const f32x2 (&b)[N]) {
    f32x2 z = mul2(a[0], b[0]);
#pragma unroll
    for (int k = 1; k < N; ++k) z = fma2(a[k], b[k], z);
    return z;
}

// 2^z of both halves; results below 2^-126 are 0 (they weigh nothing next to
// the counts, which are compared with max(y, 1)).
__device__ __forceinline__ f32x2 exp2_pair(f32x2 z) {
    float a, b;
    unpair2(z, a, b);
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(a));
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(b));
    return pair2(a, b);
}

__device__ __forceinline__ f32x2 max2(f32x2 a, float b) {
    float x, y;
    unpair2(a, x, y);
    return pair2(fmaxf(x, b), fmaxf(y, b));
}

// Calls one(c) or all() for every energy range, each with its [e0, e1): the
// channel c when only one sees the range, otherwise every channel; ranges that
// no channel sees go to none().
template <class Tab, class One, class All, class None>
__device__ __forceinline__ void for_segments(const Tab &tab, One &&one, All &&all, None &&none) {
    if (tab.segs->n == 0) {
        all(0, tab.ne);
        return;
    }
#pragma unroll 1
    for (int k = 0; k < tab.segs->n; ++k) {
        const int v = tab.segs->v[k], e0 = v & 511, e1 = (v >> 9) & 511, mask = v >> 18;
        if (mask == 0)
            none(e0, e1);
        else if ((mask & (mask - 1)) == 0)
            one(__ffs(mask) - 1, e0, e1);
        else
            all(e0, e1);
    }
}

// Runtime-indexed element of a register array (c is the same for the block).
template <int CM>
__device__ __forceinline__ f32x2 pick(const f32x2 (&a)[CM], int c) {
    f32x2 v = a[0];
#pragma unroll
    for (int k = 1; k < CM; ++k)
        if (k == c) v = a[k];
    return v;
}
template <int CM>
__device__ __forceinline__ void put(f32x2 (&a)[CM], int c, f32x2 v) {
#pragma unroll
    for (int k = 0; k < CM; ++k)
        if (k == c) a[k] = v;
}

// Mean counts yb[c] = sum_E S t of both rays; with TOP also the largest exponent
// of 2 met over all energies (-log2(e) times the smallest z), from the same
// pass.
template <bool TOP, int NM, int CM>
__device__ __forceinline__ void counts2(const SpecTab<NM, CM> &tab, const f32x2 (&l)[NM], f32x2 (&yb)[CM], float &za,
                                        float &zb) {
#pragma unroll
    for (int c = 0; c < CM; ++c) yb[c] = 0ull;
    za = zb = -3.0e38f;
    auto exponent = [&](const f32x2 (&q)[NM]) {
        const f32x2 z = neglog2e(dot2(q, l));
        if constexpr (TOP) {
            float a, b;
            unpair2(z, a, b);
            za = fmaxf(za, a), zb = fmaxf(zb, b);
        }
        return z;
    };
    for_segments(
        tab,
        [&](int c, int e0, int e1) {
            f32x2 a = pick(yb, c);
#pragma unroll 4
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s;
                tab.get(e, c, q, s);
                a = fma2(s, exp2_pair(exponent(q)), a);
            }
            put(yb, c, a);
        },
        [&](int e0, int e1) {
#pragma unroll 2
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s[CM];
                tab.get(e, q, s);
                const f32x2 t = exp2_pair(exponent(q));
#pragma unroll
                for (int c = 0; c < CM; ++c) yb[c] = fma2(s[c], t, yb[c]);
            }
        },
        [&](int e0, int e1) {
            if constexpr (TOP) {
                for (int e = e0; e < e1; ++e) {
                    f32x2 q[NM], s;
                    tab.get(e, 0, q, s);
                    exponent(q);
                }
            }
        });
}

template <int NM, int CM>
__device__ __forceinline__ void counts2(const SpecTab<NM, CM> &tab, const f32x2 (&l)[NM], f32x2 (&yb)[CM]) {
    float za, zb;
    counts2<false>(tab, l, yb, za, zb);
}

// Gradient numerators gm = -sum_E Q t v, v = -sum_c S u_c (u the negated weighted
// residuals), and, with KAPPA, the curvature numerators km = sum_E Q gamma_E c_E,
// eta = sum_c S ws_c.
template <int NM, int CM, bool KAPPA>
__device__ __forceinline__ void numerators2(const SpecTab<NM, CM> &tab, const f32x2 (&l)[NM], const f32x2 (&u)[CM],
                                            const f32x2 (&ws)[CM], const f32x2 (&gam)[NM], f32x2 (&gm)[NM],
                                            f32x2 (&km)[NM]) {
#pragma unroll
    for (int m = 0; m < NM; ++m) gm[m] = km[m] = 0ull;
    auto add = [&](const f32x2 (&q)[NM], f32x2 nv, f32x2 eta) {
        const f32x2 t = exp2_pair(neglog2e(dot2(q, l))), tv = mul2(t, nv);
#pragma unroll
        for (int m = 0; m < NM; ++m) gm[m] = fma2(q[m], tv, gm[m]);   // Q (-t v)
        if constexpr (KAPPA) {
            const f32x2 nrho = fma2(eta, t, nv), uh = max2(t, 1.f);
            const f32x2 cE = max2(mul2(sub2(mul2(add2(eta, eta), uh), nrho), uh), 0.f);
            const f32x2 w = mul2(dot2(q, gam), cE);
#pragma unroll
            for (int m = 0; m < NM; ++m) km[m] = fma2(q[m], w, km[m]);
        }
    };
    for_segments(
        tab,
        [&](int c, int e0, int e1) {
            const f32x2 uc = pick(u, c), wc = KAPPA ? pick(ws, c) : 0ull;
#pragma unroll 4
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s;
                tab.get(e, c, q, s);
                add(q, mul2(s, uc), KAPPA ? mul2(s, wc) : 0ull);
            }
        },
        [&](int e0, int e1) {
#pragma unroll 4
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s[CM];
                tab.get(e, q, s);
                add(q, dot2(s, u), KAPPA ? dot2(s, ws) : 0ull);
            }
        },
        [](int, int) {});
}

// Counts at l and their first two derivatives along -ndir, and the
// largest exponent of 2 met (-log2(e) times the smallest z), all energies.
template <int NM, int CM>
__device__ __forceinline__ void line2(const SpecTab<NM, CM> &tab, const f32x2 (&l)[NM], const f32x2 (&ndir)[NM],
                                      f32x2 (&yb)[CM], f32x2 (&d1)[CM], f32x2 (&d2)[CM], float &za, float &zb) {
#pragma unroll
    for (int c = 0; c < CM; ++c) yb[c] = d1[c] = d2[c] = 0ull;
    za = zb = -3.0e38f;
    auto exponent = [&](const f32x2 (&q)[NM]) {
        const f32x2 z = neglog2e(dot2(q, l));
        float a, b;
        unpair2(z, a, b);
        za = fmaxf(za, a), zb = fmaxf(zb, b);
        return z;
    };
    for_segments(
        tab,
        [&](int c, int e0, int e1) {
            f32x2 a = pick(yb, c), b = pick(d1, c), d = pick(d2, c);
#pragma unroll 4
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s;
                tab.get(e, c, q, s);
                const f32x2 t = exp2_pair(exponent(q)), dz = dot2(q, ndir), tdz = mul2(t, dz);
                a = fma2(s, t, a);
                b = fma2(s, tdz, b);
                d = fma2(s, mul2(tdz, dz), d);
            }
            put(yb, c, a), put(d1, c, b), put(d2, c, d);
        },
        [&](int e0, int e1) {
#pragma unroll 4
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s[CM];
                tab.get(e, q, s);
                const f32x2 t = exp2_pair(exponent(q)), dz = dot2(q, ndir), tdz = mul2(t, dz), td2 = mul2(tdz, dz);
#pragma unroll
                for (int c = 0; c < CM; ++c) {
                    yb[c] = fma2(s[c], t, yb[c]);
                    d1[c] = fma2(s[c], tdz, d1[c]);
                    d2[c] = fma2(s[c], td2, d2[c]);
                }
            }
        },
        [&](int e0, int e1) {
            for (int e = e0; e < e1; ++e) {
                f32x2 q[NM], s;
                tab.get(e, 0, q, s);
                exponent(q);
            }
        });
}

// Counts at l + alpha_k dir for K steps alpha_k at once (the exponents are
// formed from those of l and dir, once per energy), and the largest exponents.
template <int NM, int CM, int K>
__device__ __forceinline__ void candidates2(const SpecTab<NM, CM> &tab, const f32x2 (&l)[NM], const f32x2 (&dir)[NM],
                                            const float *alpha, f32x2 (&yb)[K][CM], float (&za)[K], float (&zb)[K]) {
    f32x2 al[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        al[k] = pair2(alpha[k], alpha[k]);
        za[k] = zb[k] = -3.0e38f;
#pragma unroll
        for (int c = 0; c < CM; ++c) yb[k][c] = 0ull;
    }
#pragma unroll 1
    for (int e = 0; e < tab.ne; ++e) {
        f32x2 q[NM], s[CM];
        tab.get(e, q, s);
        const f32x2 z0 = neglog2e(dot2(q, l)), z1 = neglog2e(dot2(q, dir));
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const f32x2 z = fma2(al[k], z1, z0);
            float a, b;
            unpair2(z, a, b);
            za[k] = fmaxf(za[k], a), zb[k] = fmaxf(zb[k], b);
            const f32x2 t = exp2_pair(z);
#pragma unroll
            for (int c = 0; c < CM; ++c) yb[k][c] = fma2(s[c], t, yb[k][c]);
        }
    }
}

// Two rays of one thread: i and i + blockDim.x (both loads of a warp
// coalesced whatever the alignment); past the end the last ray again, with
// nothing stored and a zero weight.
struct RayPair {
    int64_t a, b;
    bool va, vb;
    __device__ __forceinline__ RayPair(int64_t base, int64_t n) {
        a = base + threadIdx.x, b = a + blockDim.x;
        va = a < n, vb = b < n;
        if (!va) a = n - 1;
        if (!vb) b = n - 1;
    }
    __device__ __forceinline__ f32x2 load(const float *__restrict__ p) const { return pair2(__ldg(p + a), __ldg(p + b)); }
    __device__ __forceinline__ void store(float *__restrict__ p, f32x2 v) const {
        float x, y;
        unpair2(v, x, y);
        if (va) p[a] = x;
        if (vb) p[b] = y;
    }
};

// Two consecutive-row rays of one thread for the row-coupled kernels: positions
// t = threadIdx.x and + blockDim.x of an extended segment that starts at ray
// `first`; rays outside [0, n) are invalid (clamped for loads, zero counts).
struct SegPair {
    int t[2], j[2];
    int64_t i[2];
    bool valid[2];
    __device__ __forceinline__ SegPair(int64_t first, int64_t n, int row) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            t[h] = threadIdx.x + h * blockDim.x;
            i[h] = first + t[h];
            valid[h] = i[h] >= 0 && i[h] < n;
            if (!valid[h]) i[h] = i[h] < 0 ? 0 : n - 1;
            j[h] = (int)(i[h] % row);
        }
    }
    __device__ __forceinline__ f32x2 load(const float *__restrict__ p) const {
        return pair2(__ldg(p + i[0]), __ldg(p + i[1]));
    }
    __device__ __forceinline__ void put_shared(float *__restrict__ p, f32x2 v) const {
        float a, b;
        unpair2(v, a, b);
        p[t[0]] = valid[0] ? a : 0.f;
        p[t[1]] = valid[1] ? b : 0.f;
    }
};

template <int NM, int CM, bool KAPPA>
__global__ void __launch_bounds__(kModelThreads)
    model_grad_kernel(const __grid_constant__ SpecDev sp, int64_t n_rays, const float *__restrict__ l,
                      const float *__restrict__ y, const float *__restrict__ gamma, float *__restrict__ g, float *__restrict__ kappa,
                      dfloat *__restrict__ partials) {
    extern __shared__ float4 spec_smem4[];
    const int64_t step = (int64_t)gridDim.x * 2 * blockDim.x;
    int64_t base = (int64_t)blockIdx.x * 2 * blockDim.x;
    RayPair r(base, n_rays);
    f32x2 lm[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) lm[m] = r.load(l + m * n_rays);   // on its way while the table is built
    SpecTab<NM, CM> tab;
    tab.load(sp, spec_smem4);
    const int nc = sp.nc;
    dfloat obj{0.f, 0.f};
    while (base < n_rays) {
        f32x2 yb[CM], u[CM], ws[CM];
        counts2(tab, lm, yb);
#pragma unroll
        for (int c = 0; c < CM; ++c) {
            u[c] = ws[c] = 0ull;
            if (c < nc) {
                float ya, yy, ba, bb;
                unpair2(r.load(y + c * n_rays), ya, yy);
                unpair2(yb[c], ba, bb);
                const float wa = 1.f / fmaxf(ya, 1.f), wb = 1.f / fmaxf(yy, 1.f), ra = ba - ya, rb = bb - yy;
                if (r.va) df_add(obj, 0.5f * (wa * ra) * ra);
                if (r.vb) df_add(obj, 0.5f * (wb * rb) * rb);
                u[c] = pair2(-wa * ra, -wb * rb);
                ws[c] = pair2(wa * tab.sig[c], wb * tab.sig[c]);
            }
        }
        if (g || KAPPA) {
            f32x2 gm[NM], km[NM], gam[NM];
#pragma unroll
            for (int m = 0; m < NM; ++m) gam[m] = KAPPA ? r.load(gamma + m * n_rays) : 0ull;
            numerators2<NM, CM, KAPPA>(tab, lm, u, ws, gam, gm, km);
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                if (g) r.store(g + m * n_rays, gm[m]);
                if (KAPPA) r.store(kappa + m * n_rays, km[m]);
            }
        }
        base += step;
        if (base >= n_rays) break;
        r = RayPair(base, n_rays);
#pragma unroll
        for (int m = 0; m < NM; ++m) lm[m] = r.load(l + m * n_rays);
    }
    dfloat v[1] = {obj};
    block_sum_store<1>(v, partials);
}

template <int NM, int CM, int MODE>
__global__ void __launch_bounds__(kModelThreads)
    ls_fused_kernel(const __grid_constant__ SpecDev sp, int64_t n_rays, const float *__restrict__ l,
                    const float *__restrict__ q, const float *__restrict__ y, DevLS *ls, LsCfg cfg, int last, dfloat *__restrict__ partials) {
    if (MODE == 1 && ls->done) return;  // same value for every block
    extern __shared__ float4 spec_smem4[];
    const int64_t step = (int64_t)gridDim.x * 2 * blockDim.x;
    int64_t base = (int64_t)blockIdx.x * 2 * blockDim.x;
    RayPair r(base, n_rays);
    f32x2 lm[NM], qm[NM];   // on their way while the table is built
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        qm[m] = r.load(q + m * n_rays);
        lm[m] = r.load(l + m * n_rays);
    }
    const float alpha = MODE == 0 ? (float)ls->alpha : 0.f;
    auto advance = [&] {
        base += step;
        if (base >= n_rays) return false;
        r = RayPair(base, n_rays);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            qm[m] = r.load(q + m * n_rays);
            lm[m] = r.load(l + m * n_rays);
        }
        return true;
    };
    SpecTab<NM, CM> tab;
    tab.load(sp, spec_smem4);
    const int nc = sp.nc;
    const int nh = cfg.n_halve < kMaxHalve ? cfg.n_halve : kMaxHalve;
    const float z_lim = cfg.z_min * -kLog2e;   // exponents above it leave the domain
    constexpr int NACC = MODE == 0 ? 4 : 2 * kMaxHalve;
    dfloat acc[NACC];
#pragma unroll
    for (int k = 0; k < NACC; ++k) acc[k] = dfloat{0.f, 0.f};
    if constexpr (MODE == 0) {
        const f32x2 alpha2 = pair2(alpha, alpha);
        do {
            f32x2 la[NM], nq[NM], yb[CM], d1[CM], d2[CM];
            float za, zb;
#pragma unroll
            for (int m = 0; m < NM; ++m) la[m] = fma2(alpha2, qm[m], lm[m]), nq[m] = sub2(0ull, qm[m]);
            line2(tab, la, nq, yb, d1, d2, za, zb);
            float f[2] = {0.f, 0.f}, f1[2] = {0.f, 0.f}, f2[2] = {0.f, 0.f};
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (c < nc) {
                    float yv[2], b[2], e1[2], e2[2];
                    unpair2(r.load(y + c * n_rays), yv[0], yv[1]);
                    unpair2(yb[c], b[0], b[1]);
                    unpair2(d1[c], e1[0], e1[1]);
                    unpair2(d2[c], e2[0], e2[1]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float w = 1.f / fmaxf(yv[h], 1.f), res = b[h] - yv[h];
                        f[h] = fmaf(0.5f * w * res, res, f[h]);
                        f1[h] = fmaf(w * res, e1[h], f1[h]);
                        f2[h] = fmaf(w, fmaf(e1[h], e1[h], res * e2[h]), f2[h]);
                    }
                }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!(h ? r.vb : r.va)) continue;
                df_add(acc[0], f[h]);
                df_add(acc[1], f1[h]);
                df_add(acc[2], f2[h]);
                if (!((h ? zb : za) <= z_lim)) df_add(acc[3], 1.f);
            }
        } while (advance());
        block_sum_store<4>(acc, partials);
    } else {
        const double a0 = ls->best_a;
        float alphas[kMaxHalve];
        double ak = a0;
#pragma unroll
        for (int k = 0; k < kMaxHalve; ++k) {
            ak *= 0.5;
            alphas[k] = (float)ak;
        }
        do {
            constexpr int K = CM <= 2 ? 4 : (CM == 4 ? 2 : 1);   // candidates whose counts fit in registers
#pragma unroll
            for (int k0 = 0; k0 < kMaxHalve; k0 += K) {
                if (k0 >= nh) break;
                f32x2 yb[K][CM];
                float za[K], zb[K];
                candidates2<NM, CM, K>(tab, lm, qm, alphas + k0, yb, za, zb);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    float f[2] = {0.f, 0.f};
#pragma unroll
                    for (int c = 0; c < CM; ++c)
                        if (c < nc) {
                            float yv[2], b[2];
                            unpair2(r.load(y + c * n_rays), yv[0], yv[1]);
                            unpair2(yb[k][c], b[0], b[1]);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const float res = b[h] - yv[h];
                                f[h] = fmaf(0.5f / fmaxf(yv[h], 1.f) * res, res, f[h]);
                            }
                        }
                    if (r.va) {
                        df_add(acc[k0 + k], f[0]);
                        if (!(za[k] <= z_lim)) df_add(acc[kMaxHalve + k0 + k], 1.f);
                    }
                    if (r.vb) {
                        df_add(acc[k0 + k], f[1]);
                        if (!(zb[k] <= z_lim)) df_add(acc[kMaxHalve + k0 + k], 1.f);
                    }
                }
            }
        } while (advance());
        block_sum_store<NACC>(acc, partials);
    }
    if (!last_block_arrive(&ls->ticket)) return;
    const int nb = gridDim.x;
    if constexpr (MODE == 0) {
        double sums[4];
        block_sum_partials_k<4>(partials, nb, sums);
        if (threadIdx.x == 0) {
            ls_newton_control(ls, sums[0], sums[1], sums[2], sums[3], last, cfg);
            ls->ticket = 0;
        }
    } else {
        double sums[2 * kMaxHalve];
        block_sum_partials_k<2 * kMaxHalve>(partials, nb, sums);
        if (threadIdx.x == 0) {
            ls_halve_control(ls, sums, sums + kMaxHalve, nh);
            ls->ticket = 0;
        }
    }
}

// ---------------------------------------------------------------- blur
// With a detector blur B in the outer operator (B S, Eq. 1) the mean counts
// of a ray mix the unblurred counts of its row neighbours, and the SPS
// quantities of Eqs. 8 and 10 become, per ray i and energy E,
//   eta = sum_c S[c][E] sigma_c [B^T (w_c .* B 1)]_i
//   rho = sum_c S[c][E] [B^T (w_c .* r_c)]_i - eta t_E,   r = B S t - y.
// The blurred path runs in passes: unblurred counts per ray, then the
// blurred residual and its weights, then the numerators from B^T of those.

// [B v]_i (dir = +1) or [B^T v]_i (dir = -1), one channel, within the row.
__device__ __forceinline__ float blur_at(const BlurDev &B, const float *__restrict__ v, int64_t i, int dir) {
    const int j = (int)(i % B.row);
    float s = 0.f;
    for (int k = -B.r; k <= B.r; ++k) {
        const int jj = j + dir * k;
        if (jj >= 0 && jj < B.row) s = fmaf(B.b[k + B.r], v[i + dir * k], s);
    }
    return s;
}

// (B 1)_j at row position j (rows of `row` rays).
__device__ __forceinline__ float blur_ones(const BlurDev &B, int row, int j) {
    float s = 0.f;
    for (int k = -B.r; k <= B.r; ++k)
        if (j + k >= 0 && j + k < row) s += B.b[k + B.r];
    return s;
}

// w^1/2 = max(y, 1)^-1/2 of one ray's counts.
__device__ __forceinline__ float sqrt_weight(float y) { return sqrtf(1.f / fmaxf(y, 1.f)); }

// [W v]_j for one row of cells with W = D^-1/2 C^-1 D^-1/2: v holds the
// values of consecutive cells (shared memory), tid this cell, j its position
// in the row, yc the channel's counts (global) and i this cell's ray.  C^-1 is
// (1 / (1 - a^2)) times 1 (row ends) or 1 + a^2 on the diagonal and -a next
// to it.
__device__ __forceinline__ float noise_apply(const NoiseDev &N, int row, const float *__restrict__ v, int tid, int j,
                                             const float *__restrict__ yc, int64_t i) {
    const bool lo = j > 0, hi = j + 1 < row;
    const float a = N.a;
    const float s0 = sqrt_weight(yc[i]);
    float acc = ((lo && hi) ? fmaf(a, a, 1.f) : 1.f) * s0 * v[tid];
    if (lo) acc = fmaf(-a * sqrt_weight(yc[i - 1]), v[tid - 1], acc);
    if (hi) acc = fmaf(-a * sqrt_weight(yc[i + 1]), v[tid + 1], acc);
    return s0 * acc / fmaf(-a, a, 1.f);
}

// eta weight of one channel at ray i (row position j):
// [B^T (|W| (B 1))]_i, with |W| = diag(w) without correlated noise; y is the
// channel's counts (global memory), the row's neighbours of i are read from it.
__device__ __forceinline__ float coupled_eta_weight(const SpecDev &sp, int row, const float *__restrict__ y,
                                                    int64_t i, int j) {
    const BlurDev &B = sp.blur;
    const float a = sp.noise.a;
    float s = 0.f;
    for (int k = -B.r; k <= B.r; ++k) {
        const int jj = j - k;
        if (jj < 0 || jj >= row) continue;
        const int64_t p = i - k;
        float v;
        if (a > 0.f) {
            const bool lo = jj > 0, hi = jj + 1 < row;
            const float s0 = sqrt_weight(y[p]);
            float acc = ((lo && hi) ? fmaf(a, a, 1.f) : 1.f) * s0 * blur_ones(B, row, jj);
            if (lo) acc = fmaf(a * sqrt_weight(y[p - 1]), blur_ones(B, row, jj - 1), acc);
            if (hi) acc = fmaf(a * sqrt_weight(y[p + 1]), blur_ones(B, row, jj + 1), acc);
            v = s0 * acc / fmaf(-a, a, 1.f);
        } else {
            v = blur_ones(B, row, jj) / fmaxf(y[p], 1.f);
        }
        s = fmaf(B.b[k + B.r], v, s);
    }
    return s;
}

// Data term and numerators with rays coupled along detector rows (a blur B
// in the outer operator and / or correlated noise W), in one kernel: a block
// takes segments of T = 2 blockDim - 2H rays with H = 2 rb + rn halo rays on
// each side (rb the blur radius, rn = 1 with correlated noise).
// Phase 1: unblurred counts y0 of every ray of the extended segment (shared
// memory).  Phase 2: blurred residual r = B y0 - y (rays within rb + rn of
// the segment).  Phase 2b: weighted residual qw = W r (rays within rb; with
// diagonal noise qw = w r comes with phase 2) and the data term
// 1/2 r^T W r of the segment's own rays.  Phase 3 (own rays): u_c =
// [B^T qw_c]_i replaces w_c r_c and sigma_c [B^T (|W| B 1)]_i replaces
// w_c sigma_c in the numerators, with a second pass over the energies.
// [B v] and [B^T v] at thread tid's ray from a shared-memory column of
// consecutive rays (j = the ray's position in its row of `row` rays).
__device__ __forceinline__ float blur_col(const BlurDev &Bd, int row, const float *__restrict__ col, int tid, int j) {
    float s = 0.f;
    for (int k = -Bd.r; k <= Bd.r; ++k) {
        const int jj = j + k;
        if (jj >= 0 && jj < row) s = fmaf(Bd.b[k + Bd.r], col[tid + k], s);
    }
    return s;
}

__device__ __forceinline__ float blur_colT(const BlurDev &Bd, int row, const float *__restrict__ col, int tid, int j) {
    float s = 0.f;
    for (int k = -Bd.r; k <= Bd.r; ++k) {
        const int jj = j - k;
        if (jj >= 0 && jj < row) s = fmaf(Bd.b[k + Bd.r], col[tid - k], s);
    }
    return s;
}

template <int NM, int CM, bool KAPPA>
__global__ void __launch_bounds__(kModelThreads)
    model_grad_rows_kernel(const __grid_constant__ SpecDev sp, int64_t n_rays, const float *__restrict__ l,
                           const float *__restrict__ y, const float *__restrict__ gamma, float *__restrict__ g,
                           float *__restrict__ kappa, dfloat *__restrict__ partials) {
    extern __shared__ float4 spec_smem4[];
    SpecTab<NM, CM> tab;
    tab.load(sp, spec_smem4);
    const int nc = sp.nc;
    const int B = 2 * blockDim.x;                               // rays of an extended segment
    const int rb = sp.blur.r, rn = sp.noise.a > 0.f ? 1 : 0, H = 2 * rb + rn, T = B - 2 * H;
    const int row = rb > 0 ? sp.blur.row : sp.noise.row;
    float *y0s = reinterpret_cast<float *>(reinterpret_cast<char *>(spec_smem4) + SpecTab<NM, CM>::bytes(sp.ne, nc));
    float *qws = y0s + CM * B;                                  // [CM][B] counts, weighted residuals
    float *rs = qws + CM * B;                                   // [CM][B] residuals (rn only)
    const bool grads = g || KAPPA;
    const int64_t nseg = (n_rays + T - 1) / T;
    dfloat obj{0.f, 0.f};
    for (int64_t seg = blockIdx.x; seg < nseg; seg += gridDim.x) {
        const SegPair r(seg * T - H, n_rays, row);
        f32x2 lm[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) lm[m] = r.load(l + m * n_rays);
        {
            f32x2 yb[CM];
            counts2(tab, lm, yb);
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (c < nc) r.put_shared(y0s + c * B, yb[c]);
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = r.t[h];
            if (r.valid[h] && t >= rb && t < B - rb) {
                const bool own = t >= H && t < H + T;
                float f = 0.f;
#pragma unroll
                for (int c = 0; c < CM; ++c)
                    if (c < nc) {
                        const float yc = y[(int64_t)c * n_rays + r.i[h]];
                        const float w = 1.f / fmaxf(yc, 1.f);
                        const float rr = blur_col(sp.blur, row, y0s + c * B, t, r.j[h]) - yc;
                        if (rn) {
                            rs[c * B + t] = rr;
                        } else {
                            qws[c * B + t] = w * rr;
                            f = fmaf(0.5f * w * rr, rr, f);
                        }
                    }
                if (!rn && own) df_add(obj, f);
            }
        }
        __syncthreads();
        if (rn) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = r.t[h];
                if (r.valid[h] && t >= rb + 1 && t < B - rb - 1) {
                    float f = 0.f;
#pragma unroll
                    for (int c = 0; c < CM; ++c)
                        if (c < nc) {
                            const float qv =
                                noise_apply(sp.noise, row, rs + c * B, t, r.j[h], y + (int64_t)c * n_rays, r.i[h]);
                            qws[c * B + t] = qv;
                            f = fmaf(0.5f * rs[c * B + t], qv, f);
                        }
                    if (t >= H && t < H + T) df_add(obj, f);
                }
            }
            __syncthreads();
        }
        if (grads) {
            const bool own[2] = {r.valid[0] && r.t[0] >= H && r.t[0] < H + T, r.valid[1] && r.t[1] >= H && r.t[1] < H + T};
            f32x2 gm[NM], km[NM], gam[NM], u[CM], ws[CM];
#pragma unroll
            for (int m = 0; m < NM; ++m) gam[m] = KAPPA ? r.load(gamma + m * n_rays) : 0ull;
#pragma unroll
            for (int c = 0; c < CM; ++c) {
                float uv[2] = {0.f, 0.f}, wv[2] = {0.f, 0.f};
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (c < nc && own[h]) {
                        uv[h] = -blur_colT(sp.blur, row, qws + c * B, r.t[h], r.j[h]);
                        if (KAPPA)
                            wv[h] = tab.sig[c] * coupled_eta_weight(sp, row, y + (int64_t)c * n_rays, r.i[h], r.j[h]);
                    }
                u[c] = pair2(uv[0], uv[1]);
                ws[c] = pair2(wv[0], wv[1]);
            }
            numerators2<NM, CM, KAPPA>(tab, lm, u, ws, gam, gm, km);
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                float a[2];
                if (g) {
                    unpair2(gm[m], a[0], a[1]);
                    if (own[0]) g[m * n_rays + r.i[0]] = a[0];
                    if (own[1]) g[m * n_rays + r.i[1]] = a[1];
                }
                if (KAPPA) {
                    unpair2(km[m], a[0], a[1]);
                    if (own[0]) kappa[m * n_rays + r.i[0]] = a[0];
                    if (own[1]) kappa[m * n_rays + r.i[1]] = a[1];
                }
            }
        }
        __syncthreads();
    }
    if (partials) {
        dfloat v[1] = {obj};
        block_sum_store<1>(v, partials);
    }
}

// Line search with rays coupled along detector rows (blur and / or
// correlated noise), one kernel per evaluation: a block takes segments of
// T = 2 blockDim - 2H consecutive rays plus H = rb + rn halo rays on each side.
// Every thread evaluates the unblurred counts of two rays of the extended
// segment (and, for the Newton evaluation, their first two alpha-derivatives)
// into shared memory; the rays within rn of the segment blur them along their
// row; the segment's own rays then add the data terms (with correlated noise
// through W applied to the blurred residuals and derivatives of their row
// neighbours) and count the rays that leave the domain z >= z_min.  Partials
// and the last block's control are those of ls_fused_kernel.
template <int NM, int CM, int MODE>
__global__ void __launch_bounds__(kModelThreads)
    ls_rows_kernel(const __grid_constant__ SpecDev sp, int64_t n_rays, const float *__restrict__ l,
                   const float *__restrict__ q, const float *__restrict__ y, DevLS *ls, LsCfg cfg, int last,
                   dfloat *__restrict__ partials) {
    if (MODE == 1 && ls->done) return;  // same value for every block
    extern __shared__ float4 spec_smem4[];
    SpecTab<NM, CM> tab;
    tab.load(sp, spec_smem4);
    const int nc = sp.nc;
    const float z_lim = cfg.z_min * -kLog2e;
    // [NV][CM][B] with NV = 3 values per channel and ray (mode 0) or 1
    float *buf = reinterpret_cast<float *>(reinterpret_cast<char *>(spec_smem4) + SpecTab<NM, CM>::bytes(sp.ne, nc));
    const int B = 2 * blockDim.x;
    const int rb = sp.blur.r, rn = sp.noise.a > 0.f ? 1 : 0, H = rb + rn, T = B - 2 * H;
    const int row = rb > 0 ? sp.blur.row : sp.noise.row;
    const int64_t nseg = (n_rays + T - 1) / T;
    const int nh = cfg.n_halve < kMaxHalve ? cfg.n_halve : kMaxHalve;
    constexpr int NACC = MODE == 0 ? 4 : 2 * kMaxHalve;
    dfloat acc[NACC];
#pragma unroll
    for (int k = 0; k < NACC; ++k) acc[k] = dfloat{0.f, 0.f};
    float alphas[kMaxHalve];
    {
        double ak = MODE == 0 ? 0.0 : ls->best_a;
#pragma unroll
        for (int k = 0; k < kMaxHalve; ++k) {
            ak *= 0.5;
            alphas[k] = (float)ak;
        }
    }
    const float alpha = MODE == 0 ? (float)ls->alpha : 0.f;
    for (int64_t seg = blockIdx.x; seg < nseg; seg += gridDim.x) {
        const SegPair r(seg * T - H, n_rays, row);
        f32x2 lm[NM], qm[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            qm[m] = r.load(q + m * n_rays);
            lm[m] = r.load(l + m * n_rays);
        }
#pragma unroll
        for (int k = 0; k < (MODE == 0 ? 1 : kMaxHalve); ++k) {
            if (MODE == 1 && k >= nh) break;  // same for every thread
            float ze[2] = {-3.0e38f, -3.0e38f};
            {
                const float ak = MODE == 0 ? alpha : alphas[k];
                f32x2 la[NM], v0[CM], v1[CM], v2[CM];
#pragma unroll
                for (int m = 0; m < NM; ++m) la[m] = fma2(pair2(ak, ak), qm[m], lm[m]);
                if constexpr (MODE == 0) {
                    f32x2 nq[NM];
#pragma unroll
                    for (int m = 0; m < NM; ++m) nq[m] = sub2(0ull, qm[m]);
                    line2(tab, la, nq, v0, v1, v2, ze[0], ze[1]);
                } else {
                    counts2<true>(tab, la, v0, ze[0], ze[1]);
                }
#pragma unroll
                for (int c = 0; c < CM; ++c)
                    if (c < nc) {
                        r.put_shared(buf + c * B, v0[c]);
                        if (MODE == 0) {
                            r.put_shared(buf + (CM + c) * B, v1[c]);
                            r.put_shared(buf + (2 * CM + c) * B, v2[c]);
                        }
                    }
            }
            __syncthreads();
            // blurred residual and derivatives at the rays within rn of the
            // segment (registers first: the neighbours still read buf)
            float r0[2][CM], r1[2][CM], r2[2][CM], sw[2][CM];
            bool own[2], near[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = r.t[h];
                own[h] = r.valid[h] && t >= H && t < H + T;
                near[h] = r.valid[h] && t >= rb && t < B - rb;   // blurred values needed here
                if (own[h] && !(ze[h] <= z_lim)) df_add(acc[MODE == 0 ? 3 : kMaxHalve + k], 1.f);
#pragma unroll
                for (int c = 0; c < CM; ++c) {
                    r0[h][c] = r1[h][c] = r2[h][c] = 0.f;
                    sw[h][c] = 0.f;
                    if (c < nc && near[h]) {
                        const float yc = y[(int64_t)c * n_rays + r.i[h]];
                        sw[h][c] = 1.f / fmaxf(yc, 1.f);
                        r0[h][c] = blur_col(sp.blur, row, buf + c * B, t, r.j[h]) - yc;
                        if (MODE == 0) {
                            r1[h][c] = blur_col(sp.blur, row, buf + (CM + c) * B, t, r.j[h]);
                            r2[h][c] = blur_col(sp.blur, row, buf + (2 * CM + c) * B, t, r.j[h]);
                        }
                    }
                }
            }
            if (rn) {
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (near[h])
#pragma unroll
                        for (int c = 0; c < CM; ++c)
                            if (c < nc) {
                                buf[c * B + r.t[h]] = r0[h][c];
                                if (MODE == 0) buf[(CM + c) * B + r.t[h]] = r1[h][c];
                            }
                __syncthreads();
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!own[h]) continue;
                float f = 0.f, f1 = 0.f, f2 = 0.f;
#pragma unroll
                for (int c = 0; c < CM; ++c)
                    if (c < nc) {
                        // W r and W r' at this ray (diagonal: w r, w r')
                        float wr, wd;
                        if (rn) {
                            const float *yc = y + (int64_t)c * n_rays;
                            wr = noise_apply(sp.noise, row, buf + c * B, r.t[h], r.j[h], yc, r.i[h]);
                            wd = MODE == 0 ? noise_apply(sp.noise, row, buf + (CM + c) * B, r.t[h], r.j[h], yc, r.i[h])
                                           : 0.f;
                        } else {
                            wr = sw[h][c] * r0[h][c];
                            wd = sw[h][c] * r1[h][c];
                        }
                        f = fmaf(0.5f * r0[h][c], wr, f);
                        if (MODE == 0) {
                            f1 = fmaf(r1[h][c], wr, f1);
                            f2 = fmaf(r1[h][c], wd, fmaf(r2[h][c], wr, f2));
                        }
                    }
                if (MODE == 0) {
                    df_add(acc[0], f);
                    df_add(acc[1], f1);
                    df_add(acc[2], f2);
                } else {
                    df_add(acc[k], f);
                }
            }
            __syncthreads();
        }
    }
    block_sum_store<NACC>(acc, partials);
    if (!last_block_arrive(&ls->ticket)) return;
    const int nb = gridDim.x;
    if constexpr (MODE == 0) {
        double sums[4];
        block_sum_partials_k<4>(partials, nb, sums);
        if (threadIdx.x == 0) {
            ls_newton_control(ls, sums[0], sums[1], sums[2], sums[3], last, cfg);
            ls->ticket = 0;
        }
    } else {
        double sums[2 * kMaxHalve];
        block_sum_partials_k<2 * kMaxHalve>(partials, nb, sums);
        if (threadIdx.x == 0) {
            ls_halve_control(ls, sums, sums + kMaxHalve, nh);
            ls->ticket = 0;
        }
    }
}

}  // namespace
}  // namespace psps
