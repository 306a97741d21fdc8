// Per-ray spectral forward model, PWLS data term, SPS numerators and
// line-search terms (model.cu).
#pragma once
#include "common.cuh"
#include "ls.cuh"

namespace psps {

// Detector blur of the outer operator (B S): [B v]_i = sum_k b[k + r] v_{i+k},
// k = -r..r, within rows of `row` consecutive rays (zero past the row ends).
struct BlurDev {
    int r = 0, row = 1;
    float b[7] = {};
};

// Correlated noise: W = Sigma_y^-1 = D^-1/2 C^-1 D^-1/2 with the tridiagonal
// inverse of the row correlation C[j][k] = a^|j-k| (a = 0: diagonal).
struct NoiseDev {
    float a = 0.f;
    int row = 1;
};

// Energy ranges between which the set of channels that see an energy (S > 0)
// changes: photon-counting channels each see their own range, the channels of
// a dual-kVp scan overlap only up to the lower voltage.  A channel's terms
// outside its set are exact zeros, so leaving them out changes no sum.  n = 0:
// one range, every channel.
constexpr int kMaxSeg = 12;
struct SpecSegs {
    int n = 0;
    int v[kMaxSeg] = {};   // first | end << 9 | channel mask << 18
};

struct SpecDev {
    int nm, ne, nc;
    const float *qs;  // Q[ne][nm], S[nc][ne], sigma[nc] (sigma_c = sum_E S[c][E])
    BlurDev blur;     // r = 0: no blur (b[0] = 1, the identity)
    NoiseDev noise;
    SpecSegs segs;
};

inline SpecDev spec_dev(const mbmd_spectrum *s) {
    SpecDev d{s->n_mat, s->n_energy, s->n_chan, s->qs.p, {}, {}, {}};
    for (int e = 0; e < s->n_energy; ++e) {
        int mask = 0;
        for (int c = 0; c < s->n_chan; ++c) mask |= (float)s->hS[c * s->n_energy + e] != 0.f ? 1 << c : 0;
        if (d.segs.n && d.segs.v[d.segs.n - 1] >> 18 == mask) {
            d.segs.v[d.segs.n - 1] += 1 << 9;
        } else if (d.segs.n == kMaxSeg) {
            d.segs.n = 0;   // too many ranges: one, every channel
            break;
        } else {
            d.segs.v[d.segs.n++] = e | (e + 1) << 9 | mask << 18;
        }
    }
    d.blur.r = s->blur_r;
    d.blur.row = s->blur_row;
    for (int k = 0; k < 7; ++k) d.blur.b[k] = s->blur_b[k];
    if (d.blur.r == 0) d.blur.b[0] = 1.f;
    d.noise.a = s->noise_a;
    d.noise.row = s->noise_row;
    return d;
}

// Rays couple along detector rows (a blur or correlated noise): the model
// and line-search kernels then work on row segments with halo rays.
inline bool row_coupled(const SpecDev &sp) { return sp.blur.r > 0 || sp.noise.a > 0.f; }

constexpr int kModelThreads = 128;
constexpr int kModelMaxBlocks = 2048;  // partial sums per block at most

// Two rays per thread at a time, a grid-stride loop over steps of 256 rays by
// b blocks per SM: of b = 8 .. 5 (enough warps to keep the FP32 pipe busy) the
// one that fills the last step best, since a nearly empty last step costs its
// whole latency (720 x 888 rays, 2 materials, 121 energies, 2 channels: 152 us
// for the line search with b = 8, whose third step holds 5 % of the blocks,
// 147 with b = 6; 3 materials, 4 channels 257 and 236).
inline int model_blocks(int64_t n) {
    const int64_t steps = cdiv(n, 2 * kModelThreads);
    static_assert(152 * 8 <= kModelMaxBlocks, "partials");
    // small scans: a block for every segment of the row-coupled kernels too,
    // whose halos take up to 14 of a step's rays (a block with two segments
    // takes twice as long as all others: 20000 blurred rays, 6 channels 66 us for
    // the gradient, 59 with a block each)
    const int64_t segs = cdiv(n, 2 * kModelThreads - 14);
    if (segs <= 152 * 8) return (int)(segs < 1 ? 1 : segs);
    int best = 8;
    double fill = 0.0;
    for (int b = 8; b >= 5; --b) {
        const double s = (double)steps / (152.0 * b), f = s - (double)(int64_t)s;
        const double last = (f == 0.0 ? 1.0 : f);
        if (s < 32.0 && last > fill + 0.01) best = b, fill = last;
    }
    return 152 * best;
}

// data term partials (1 per block); g, kappa optional ([nm][n_rays]).
// gamma: per-ray gamma_m = [A |M| 1]_m ([nm][n_rays]) for kappa.  With a
// detector blur or correlated noise the same quantities come from row
// segments with halos (one kernel, no scratch).
mbir_status launch_model_grad(SpecDev sp, int64_t n_rays, const float *l, const float *y, const float *gamma,
                              float *g, float *kappa, dfloat *partials, int nblocks, cudaStream_t s);
// Fused line-search evaluation: mode 0 evaluates phi, phi', phi'' at
// ls->alpha and its last block runs the Newton control; mode 1 (skipped when
// the search is done) evaluates the n_halve halving candidates at once and
// its last block picks the step.  partials: 2 kMaxHalve per block.  With a
// detector blur or correlated noise the same evaluation runs on row segments
// with halos (one kernel, no scratch).
mbir_status launch_ls_fused(SpecDev sp, int64_t n_rays, const float *l, const float *q, const float *y, DevLS *ls,
                            LsCfg cfg, int mode, int last, dfloat *partials, int nblocks, cudaStream_t s);
// ybar = B S exp(-Q l); with a blur, y0 ([n_chan][n_rays]) holds the unblurred
// counts.
mbir_status launch_forward_model(SpecDev sp, int64_t n_rays, const float *l, float *ybar, cudaStream_t s,
                                 float *y0 = nullptr);
// Per-ray Fisher blocks F_i = Q^T D S^T W S D Q (upper triangle, packed
// [nm(nm+1)/2][n_rays]) with D = y / I0 (one energy/channel) or the water fit.
mbir_status launch_fisher_blocks(const mbmd_spectrum *spec, int64_t n_rays, const float *y, float *F,
                                 cudaStream_t s);

}  // namespace psps
