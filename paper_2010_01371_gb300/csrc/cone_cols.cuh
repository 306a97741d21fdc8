// Detector-column view of the cone-beam projector, shared by cone.cu (set-up,
// general kernels) and cone_cols.cu (the column kernels).
//
// The detector rows run along z, so all rays of one detector column (view v,
// column iu) lie in one plane through the source that contains the z axis
// direction.  On plane i of its driving axis a (t = i - c_a, c_a the middle):
//   in-plane coordinate  b = b0 + t db                    (same for every row)
//   height               z = (row offset) (q0 + t dq)     (voxels, from the middle)
// col[v * n_u + iu] = (b0 - 1/2 - (n_b >> 1), db, q0, dq) and
// colw = (pixel size / |d_a|, bits(axis | lo << 2 | hi << 17)), [lo, hi] the
// planes on which b can lie in (-1, n_b).
#pragma once
#include "common.cuh"

namespace psps {

// Zero rows on both sides of a column of the transpose's weighted sinogram.
constexpr int kRowPad = 8;

// Height of the middle of the volume as index less 1/2, relative to n / 2.
__host__ __device__ inline float cone_z_offset(int nz) { return 0.5f * (nz - 1) - 0.5f - (float)(nz >> 1); }

__device__ __forceinline__ void decode_col(float2 W, int &axis, int &lo, int &hi) {
    const int bits = __float_as_int(W.y);
    axis = bits & 3;
    lo = (bits >> 2) & 0x7fff;
    hi = (bits >> 17) & 0x7fff;
}

// Ray weight (pixel size) |d| / |d_a| at detector offsets u, w.
__device__ __forceinline__ float cone_weight(const mbir_geometry &g, float2 W, float u, float w) {
    const float sdd = (float)g.sdd;
    return W.x * sqrtf(fmaf(w, w, fmaf(u, u, sdd * sdd)));
}

// Packed copies of x[m][z][y][x] for each driving axis a, materials innermost
// with stride P (1, 2 or 4), each plane with kPad zero cells on both sides of
// b and c.  The columns' lanes run along z and read [a][b][c], c = z fastest;
// the general kernel's lanes run along the detector row and read [a][c][b].
constexpr int kPad = 2;

template <int NM>
struct CPack;
template <>
struct CPack<1> {
    using T = float;
    __device__ static void get(const T &v, float (&o)[1]) { o[0] = v; }
};
template <>
struct CPack<2> {
    using T = float2;
    __device__ static void get(const T &v, float (&o)[2]) { o[0] = v.x, o[1] = v.y; }
};
template <>
struct CPack<4> {
    using T = float4;
    __device__ static void get(const T &v, float (&o)[4]) { o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w; }
};

// Volume copies [a][c][b] of nm materials (P floats per cell) into the plan's
// scratch; the copy of the z-driven rays only when z_too.
mbir_status cone_pack_rows(mbir_plan *p, const float *x, int nm, int P, bool z_too, cudaStream_t s);
// Whether the column forward pays for P materials (p->cols given).
bool cone_cols_forward(const mbir_geometry &g, int P);
// The column kernels' rules and buffers, decided once per plan.
mbir_status cone_cols_setup(mbir_plan *p);
// l[m] = A x[m] for nm <= 4 materials; x[c] (+)= A^T sino[c] for nc <= 4
// channels.  Only for plans with p->cols / p->col_rows > 0.
mbir_status project_cone_cols(mbir_plan *p, const float *x, float *l, int nm, cudaStream_t s);
mbir_status backproject_cone_cols(mbir_plan *p, const float *sino, float *x, int nc, int accumulate, cudaStream_t s);

}  // namespace psps
