// The projector pair and the data agents of plans whose detector or volume is too
// thin for lanes along the detector rows and along z (projector.cu): lanes along
// the detector columns and along x, volumes as planes of z-pairs.
//
// Same model and per-ray arithmetic: A equals the other layout's bit for bit, A^T to
// rounding.  What decides between the two is in choose_routes (projector.cu).  At
// 256^2 x 4 voxels, 384 columns, 48 views per frame, these kernels against the lines':
//   nz = 1, nv = 1:   A 118 against 690 us, A^T 281 against 830, two CG steps 1.24 against 4.8 ms
//   nz = 8, nv = 8:   265 against 705, 451 against 820, 2.25 against 4.8 ms
//   nz = 16, nv = 33: 555 against 895, 1137 against 1370, 5.2 against 6.9 ms
// The pairs cost 16 bytes per voxel.
#include <math.h>

#include <algorithm>

#include "projector.cuh"

namespace msf {

// ------------------------------------------------------------------ z-paired copies

// Per frame and z-slice, the two copies of a volume v that the forward reads:
// py[z][y][x] = (v(z, y, x), v(z + 1, y, x)) and px[z][x][y], the same pairs
// transposed (x-major rays read y-contiguous data), with v(nz, ., .) = 0, so
// that a ray's four bilinear taps are two 8-byte loads.
// FUSED: v = r + beta_t p (the CG direction update) with p = in; v is also
// written to pnext (a different buffer: neighbouring slices still read p).
template <bool FUSED>
__global__ void pair_kernel(const float* __restrict__ in, float2* __restrict__ px, float2* __restrict__ py,
                            const float* __restrict__ r, float* __restrict__ pnext, const double* __restrict__ beta,
                            int nx, int ny, int nz) {
    __shared__ float2 tile[32][33];
    const int slice = blockIdx.z;             // t * nz + z
    const int t = slice / nz, z = slice % nz;
    const size_t plane = (size_t)nx * ny;
    const size_t base = (size_t)slice * plane;
    const bool up = z + 1 < nz;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    float bt = 0.0f;
    if (FUSED) bt = (float)beta[t];
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int x = x0 + threadIdx.x, y = y0 + k;
        if (x < nx && y < ny) {
            const size_t i = base + (size_t)y * nx + x;
            float lo, hi = 0.0f;
            if (FUSED) {
                lo = __fmaf_rn(bt, in[i], r[i]);
                if (up) hi = __fmaf_rn(bt, in[i + plane], r[i + plane]);
                pnext[i] = lo;
            } else {
                lo = in[i];
                if (up) hi = in[i + plane];
            }
            const float2 v = make_float2(lo, hi);
            py[i] = v;
            tile[k][threadIdx.x] = v;
        }
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int y = y0 + threadIdx.x, x = x0 + k;
        if (x < nx && y < ny) px[base + (size_t)x * ny + y] = tile[threadIdx.x][k];
    }
}
// ------------------------------------------------------------------ forward

// Rays per thread of the forward: consecutive detector rows of one column,
// which share the column's in-plane crossing (f_a, its floor and weight).
constexpr int PLANES_R = 2;

// Narrows [kmin, kmax] to the planes k where f(k) = f0 + (k - cmaj) b lies in
// [lo, hi], one plane inside the exact bounds on each side (so that FP32
// rounding of f never leaves [lo, hi] inside the range).
__device__ __forceinline__ void planes_within(float f0, float b, float lo, float hi, float cmaj, float& kmin,
                                              float& kmax) {
    if (fabsf(b) > 1e-12f) {
        const float k1 = (lo - f0) / b + cmaj, k2 = (hi - f0) / b + cmaj;
        kmin = fmaxf(kmin, ceilf(fminf(k1, k2)) + 1.0f);
        kmax = fminf(kmax, floorf(fmaxf(k1, k2)) - 1.0f);
    } else if (!(f0 >= lo && f0 <= hi)) {
        kmax = kmin - 1.0f;
    }
}

// One thread per PLANES_R rays (detector rows PLANES_R*i .. PLANES_R*i + PLANES_R - 1 of one
// column); a block covers blockDim.x columns x PLANES_R*blockDim.y rows of one view
// (128 threads; the shape is chosen per plan by msf_projector_autotune).  x-major
// rays read the z-paired transposed frame px [nz][nx][ny], y-major rays the
// z-paired natural frame py [nz][ny][nx] (pair_kernel), so the minor in-plane
// axis is contiguous and each (a, z) tap pair is one 8-byte load.  Planes
// where every bilinear tap of every ray of the thread lies inside the grid run
// without bounds checks; the planes at either end check each tap.  The
// interpolation is v00 + w_a (v01 - v00) along a, then the same along z.
//   FWD_PLAIN:    out = A x
//   FWD_LAMBDA:   out = step * Lambda * (A x)
//   PLANES_RESIDUAL: out = step * Lambda * (meas - A x)
// (the CG modes write the step-weighted sinogram e' = step * e that the gather
// adjoint consumes)
// PAR (the ICD agent's projection of a group step): x is zero outside one
// voxel parity group, so an x-major ray only visits planes x = kpx (mod 2) and
// a y-major ray planes y = kpy (mod 2), and on a visited plane it loads only
// the z-pair of the minor-axis tap with the group's parity (the other is zero);
// the skipped terms are exact zeros, so the result equals the full projection
// bit for bit.
template <int MODE, bool PAR = false>
__global__ void __launch_bounds__(128) planes_fwd_kernel(
    const float2* __restrict__ px, const float2* __restrict__ py, const float4* __restrict__ col,
    float* __restrict__ out, const float* __restrict__ lam, const float* __restrict__ meas,
    ProjDims d, int kpx = 0, int kpy = 0) {
    const int iu = blockIdx.x * blockDim.x + threadIdx.x;
    const int iv0 = (blockIdx.y * blockDim.y + threadIdx.y) * PLANES_R;
    const int g = blockIdx.z;
    if (iu >= d.nu || iv0 >= d.nv) return;
    const int t = g / d.views;
    const ColParams c = load_col(col, (size_t)g * d.nu + iu);
    const bool xmaj = c.xmajor != 0.0f;
    const int nmaj = xmaj ? d.nx : d.ny, na = xmaj ? d.ny : d.nx;
    const size_t fs = (size_t)d.nx * d.ny * d.nz;
    const float2* __restrict__ vol = (xmaj ? px : py) + (size_t)t * fs;   // (v(z), v(z+1)) pairs
    const float cmaj = xmaj ? d.cx : d.cy;
    const int zs = nmaj * na;    // z stride of the frame

    RayZ rz[PLANES_R];
#pragma unroll
    for (int r = 0; r < PLANES_R; ++r) rz[r] = ray_z(c, det_v(min(iv0 + r, d.nv - 1), d), d.cz);

    // planes where some crossing can touch the grid (-1 < f < n on both minor
    // axes, one plane of margin), and the inner planes where all four taps of
    // every ray are inside (0.5 <= f <= n - 1.5)
    float klo = (float)(nmaj - 1), khi = 0.0f;
    float kin_lo = 0.0f, kin_hi = (float)(nmaj - 1);
    planes_within(c.fa_mid, c.ba, 0.5f, (float)na - 1.5f, cmaj, kin_lo, kin_hi);
#pragma unroll
    for (int r = 0; r < PLANES_R; ++r) {
        float lo = 0.0f, hi = (float)(nmaj - 1);
        const float fm[2] = {c.fa_mid, rz[r].fz_mid}, bb[2] = {c.ba, rz[r].bz};
        const float top[2] = {(float)na, (float)d.nz};
        for (int a = 0; a < 2; ++a) {
            if (fabsf(bb[a]) > 1e-12f) {
                const float k1 = (-1.0f - fm[a]) / bb[a] + cmaj, k2 = (top[a] - fm[a]) / bb[a] + cmaj;
                lo = fmaxf(lo, floorf(fminf(k1, k2)) - 1.0f);
                hi = fminf(hi, ceilf(fmaxf(k1, k2)) + 1.0f);
            } else if (!(fm[a] > -1.0f && fm[a] < top[a])) {
                hi = -1.0f;
            }
        }
        if (lo <= hi) {
            klo = fminf(klo, lo);
            khi = fmaxf(khi, hi);
        }
        planes_within(rz[r].fz_mid, rz[r].bz, 0.5f, (float)d.nz - 1.5f, cmaj, kin_lo, kin_hi);
    }
    float acc[PLANES_R];
#pragma unroll
    for (int r = 0; r < PLANES_R; ++r) acc[r] = 0.0f;
    if (klo <= khi) {
        const int K0 = (int)klo, K1 = (int)khi;
        int F0 = (int)fmaxf(kin_lo, klo), F1 = (int)fminf(kin_hi, khi);
        if (F0 > F1) F0 = K1 + 1, F1 = K1;

        // one plane with every tap checked against the grid
        auto checked = [&](int k) {
            const float tk = __fsub_rn((float)k, cmaj);
            const float fa = __fmaf_rn(tk, c.ba, c.fa_mid);
            const float a0f = floorf(fa);
            const float wa1 = __fsub_rn(fa, a0f);
            const int ia = (int)a0f;
            const bool a_in0 = ia >= 0 && ia < na, a_in1 = ia + 1 >= 0 && ia + 1 < na;
#pragma unroll
            for (int r = 0; r < PLANES_R; ++r) {
                const float fz = __fmaf_rn(tk, rz[r].bz, rz[r].fz_mid);
                const float z0f = floorf(fz);
                const float wz1 = __fsub_rn(fz, z0f);
                const int iz = (int)z0f;
                // the pair of slice iz holds taps iz and iz + 1 (0 above the
                // grid); below it (iz = -1) only the upper tap, from slice 0
                float v00 = 0.0f, v01 = 0.0f, v10 = 0.0f, v11 = 0.0f;
                if (iz >= 0 && iz < d.nz) {
                    const float2* row = vol + ((ptrdiff_t)iz * nmaj + k) * na;
                    if (a_in0) { const float2 q = __ldg(row + ia); v00 = q.x; v10 = q.y; }
                    if (a_in1) { const float2 q = __ldg(row + ia + 1); v01 = q.x; v11 = q.y; }
                } else if (iz == -1) {
                    const float2* row = vol + (ptrdiff_t)k * na;
                    if (a_in0) v10 = __ldg(row + ia).x;
                    if (a_in1) v11 = __ldg(row + ia + 1).x;
                }
                const float top = __fmaf_rn(wa1, __fsub_rn(v01, v00), v00);
                const float bot = __fmaf_rn(wa1, __fsub_rn(v11, v10), v10);
                acc[r] = __fadd_rn(acc[r], __fmaf_rn(wz1, __fsub_rn(bot, top), top));
            }
        };
        const int kp = xmaj ? kpx : kpy, ka = xmaj ? kpy : kpx;
        for (int k = K0; k < F0; ++k)
            if (!PAR || (k & 1) == kp) checked(k);
        for (int k = PAR ? F0 + ((F0 ^ kp) & 1) : F0; k <= F1; k += PAR ? 2 : 1) {
            const float tk = __fsub_rn((float)k, cmaj);
            const float fa = __fmaf_rn(tk, c.ba, c.fa_mid);
            const float a0f = floorf(fa);
            const float wa1 = __fsub_rn(fa, a0f);
            const float2* pk = vol + k * na + (int)a0f;
            const bool lo = (((int)a0f) & 1) == ka;   // PAR: the tap at a0 has the group's parity
#pragma unroll
            for (int r = 0; r < PLANES_R; ++r) {
                const float fz = __fmaf_rn(tk, rz[r].bz, rz[r].fz_mid);
                const float z0f = floorf(fz);
                const float wz1 = __fsub_rn(fz, z0f);
                const float2* p0 = pk + (ptrdiff_t)((int)z0f) * zs;
                const float2 zero = make_float2(0.0f, 0.0f);
                const float2 q0 = (!PAR || lo) ? __ldg(p0) : zero;
                const float2 q1 = (!PAR || !lo) ? __ldg(p0 + 1) : zero;
                const float v00 = q0.x, v10 = q0.y, v01 = q1.x, v11 = q1.y;
                const float top = __fmaf_rn(wa1, __fsub_rn(v01, v00), v00);
                const float bot = __fmaf_rn(wa1, __fsub_rn(v11, v10), v10);
                acc[r] = __fadd_rn(acc[r], __fmaf_rn(wz1, __fsub_rn(bot, top), top));
            }
        }
        for (int k = F1 + 1; k <= K1; ++k)
            if (!PAR || (k & 1) == kp) checked(k);
    }
#pragma unroll
    for (int r = 0; r < PLANES_R; ++r) {
        const int iv = iv0 + r;
        if (iv >= d.nv) break;
        const float val = acc[r] * rz[r].step;
        const size_t ray = ((size_t)g * d.nv + iv) * d.nu + iu;
        if (MODE == FWD_PLAIN) out[ray] = val;
        else if (MODE == FWD_LAMBDA) out[ray] = rz[r].step * (lam[ray] * val);
        else out[ray] = rz[r].step * (lam[ray] * (meas[ray] - val));
    }
}

// ------------------------------------------------------------------ adjoint (gather)

// Voxels of one z-run handled by one thread of the gather: 8, 16, 32 or 64,
// chosen per plan (default 16).

// Adds, for the rays of one view whose major axis is XMAJ, w(ray, voxel) *
// e'(ray) to the ZB accumulators of the voxel run (ix, iy, iz_lo ..
// iz_lo+ZB-1), where e' = step * e is the step-weighted sinogram.
//
// An x-major ray touches column (ix, iy) on plane k = ix when floor(f_y) is
// iy-1 or iy.  Candidate detector columns come from the exact projection of
// the segment {x = x_ix, |y - y_iy| <= voxel} (plus one column of margin); on
// a column that qualifies, the rows whose f_z(k) can fall within one voxel of
// the run follow from f_z(v) = c_z + v (c1 + tk inv_dmaj).  Each ray's f_a is
// recomputed with the forward's own operations (bit for bit); f_z of row 0
// likewise, and of a row iv by one FMA from it (a few 1e-5 voxel from the
// forward's value, so the taps agree except within that distance of a voxel
// boundary, where the weights are continuous; the value depends on the ray
// alone, not on the run length the plan's autotuner picks).
// Every ray-plane crossing of the forward is visited by the two runs that hold
// its a-taps, so the work tracks the forward's.
template <bool XMAJ, int ZB>
__device__ __forceinline__ void gather_runs(const float4* __restrict__ col, const float* __restrict__ e,
                                            int g, int ix, int iy, int iz_lo, float cs, float sn,
                                            const ProjDims& d, float (*acc)[128], int tid) {
    const int kpl = XMAJ ? ix : iy;             // plane index along the major axis
    const int ia = XMAJ ? iy : ix;              // voxel index on the minor axis
    const float cmaj = XMAJ ? d.cx : d.cy;
    const float xc = (ix - d.cx) * d.vox, yc = (iy - d.cy) * d.vox;
    float u1, u2;
    if (XMAJ) {
        u1 = u_pixel(xc, yc - d.vox, cs, sn, d);
        u2 = u_pixel(xc, yc + d.vox, cs, sn, d);
    } else {
        u1 = u_pixel(xc - d.vox, yc, cs, sn, d);
        u2 = u_pixel(xc + d.vox, yc, cs, sn, d);
    }
    const int iu_lo = max(0, (int)floorf(fminf(u1, u2)) - 1);
    const int iu_hi = min(d.nu - 1, (int)ceilf(fmaxf(u1, u2)) + 1);
    const float tk = __fsub_rn((float)kpl, cmaj);
    const float inv_dv = 1.0f / d.dv;
    for (int iu = iu_lo; iu <= iu_hi; ++iu) {
        const ColParams c = load_col(col, (size_t)g * d.nu + iu);
        if ((c.xmajor != 0.0f) != XMAJ) continue;
        const float fa = __fmaf_rn(tk, c.ba, c.fa_mid);
        const float a0f = floorf(fa);
        const int a0 = (int)a0f;
        if (ia != a0 && ia != a0 + 1) continue;
        const float wa1 = __fsub_rn(fa, a0f);
        const float wa = (ia == a0) ? __fsub_rn(1.0f, wa1) : wa1;
        // rows with f_z in (iz_lo - 1, iz_lo + ZB); gz > 0 (planes lie
        // between source and detector)
        const float rgz = __fdividef(1.0f, c.c1 + tk * c.inv_dmaj);
        const float va = (iz_lo - 1 - d.cz) * rgz * inv_dv + d.cv;
        const float vb = (iz_lo + ZB - d.cz) * rgz * inv_dv + d.cv;
        const int iv_lo = max(0, (int)floorf(va) - 1);
        const int iv_hi = min(d.nv - 1, (int)ceilf(vb) + 1);
        const float* erow = e + ((size_t)g * d.nv) * d.nu + iu;
        // f_z is affine in the row: f_z(iv) = f_z(0) + iv dfz, with f_z(0) the
        // forward's crossing of detector row 0 (so a ray's value does not
        // depend on the run that evaluates it; within a few 1e-5 voxel of the
        // forward's own FP32 value)
        const RayZ rzb = ray_z(c, det_v(0, d), d.cz);
        const float fzb = __fmaf_rn(tk, rzb.bz, rzb.fz_mid);
        const float dfz = d.dv * __fmaf_rn(tk, c.inv_dmaj, c.c1);   // > 0
        // rows in [iva, ivb) have both z taps inside the run (f_z in
        // [iz_lo + 0.01, iz_lo + ZB - 1.01]); the others are checked
        const float rdfz = __fdividef(1.0f, dfz);
        const int iva = min(max((int)ceilf(((float)iz_lo + 0.01f - fzb) * rdfz), iv_lo), iv_hi + 1);
        const int ivb = min(max((int)floorf(((float)(iz_lo + ZB) - 1.01f - fzb) * rdfz) + 1, iva), iv_hi + 1);
        // explicit roundings: both loops must form a row's terms identically
        auto checked = [&](int iv) {
            const float fz = __fmaf_rn((float)iv, dfz, fzb);
            const float z0f = floorf(fz);
            const int k0 = (int)z0f - iz_lo;
            if (k0 < -1 || k0 >= ZB) return;
            const float ev = __fmul_rn(wa, __ldg(erow + (size_t)iv * d.nu));
            const float c1 = __fmul_rn(__fsub_rn(fz, z0f), ev);
            if (k0 >= 0) acc[k0][tid] = __fadd_rn(acc[k0][tid], __fsub_rn(ev, c1));
            if (k0 + 1 < ZB) acc[k0 + 1][tid] = __fadd_rn(acc[k0 + 1][tid], c1);
        };
        for (int iv = iv_lo; iv < iva; ++iv) checked(iv);
        for (int iv = iva; iv < ivb; ++iv) {
            const float fz = __fmaf_rn((float)iv, dfz, fzb);
            const float z0f = floorf(fz);
            const int k0 = min(max((int)z0f - iz_lo, 0), ZB - 2);   // in range by the choice of [iva, ivb)
            const float ev = __fmul_rn(wa, __ldg(erow + (size_t)iv * d.nu));
            const float c1 = __fmul_rn(__fsub_rn(fz, z0f), ev);
            acc[k0][tid] = __fadd_rn(acc[k0][tid], __fsub_rn(ev, c1));
            acc[k0 + 1][tid] = __fadd_rn(acc[k0 + 1][tid], c1);
        }
        for (int iv = ivb; iv <= iv_hi; ++iv) checked(iv);
    }
}

// One thread per run of ZB voxels along z; block 32 (x) x 4 (y).
// e is the step-weighted sinogram e' = step * e.
//   ADJ_PLAIN:   out = A^T e
//   ADJ_CG_INIT: r = A^T e + (v - z)/sigma^2, p = r, rr = r.r
//   ADJ_CG_Q:    q = A^T e + p/sigma^2, alpha = rr / p.q
// (at most 64 registers: eight blocks per SM, no spills)
template <int MODE, int ZB>
__global__ void __launch_bounds__(128, 8) planes_adj_kernel(
    const float4* __restrict__ col, const float2* __restrict__ trig, const int* __restrict__ vflag,
    const float* __restrict__ e, float* __restrict__ out, const float* __restrict__ a1,
    const float* __restrict__ a2, float* __restrict__ out2, CgScalars cg,
    float inv_s2, ProjDims d) {
    __shared__ float acc[ZB][128];
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int ix = blockIdx.x * 32 + threadIdx.x;
    const int iy = blockIdx.y * 4 + threadIdx.y;
    const int nzb = (d.nz + ZB - 1) / ZB;
    const int zb = blockIdx.z % nzb;
    const int t = blockIdx.z / nzb;
    const int iz_lo = zb * ZB;
    const bool inside = ix < d.nx && iy < d.ny;
#pragma unroll
    for (int k = 0; k < ZB; ++k) acc[k][tid] = 0.0f;
    if (inside) {
        for (int j = 0; j < d.views; ++j) {
            const int g = t * d.views + j;
            const float2 cs = __ldg(trig + g);
            const int fl = __ldg(vflag + g);
            if (fl & 1) gather_runs<true, ZB>(col, e, g, ix, iy, iz_lo, cs.x, cs.y, d, acc, tid);
            if (fl & 2) gather_runs<false, ZB>(col, e, g, ix, iy, iz_lo, cs.x, cs.y, d, acc, tid);
        }
    }
    double dot = 0.0;
    for (int k = 0; k < ZB; ++k) {
        const int iz = iz_lo + k;
        if (!inside || iz >= d.nz) break;
        const size_t i = (((size_t)t * d.nz + iz) * d.ny + iy) * d.nx + ix;
        const float s = acc[k][tid];
        if (MODE == ADJ_PLAIN) {
            out[i] = s;
        } else if (MODE == ADJ_CG_INIT) {   // a1 = v, a2 = z
            const float r = s + (a1[i] - a2[i]) * inv_s2;
            out[i] = r;
            out2[i] = r;
            dot += (double)r * (double)r;
        } else {                            // a1 = p
            const float p = a1[i];
            const float q = s + p * inv_s2;
            out[i] = q;
            dot += (double)p * (double)q;
        }
    }
    if (MODE != ADJ_PLAIN) {
        const double sum = block_sum_f64(dot);
        const int bpf = gridDim.x * gridDim.y * nzb;   // blocks per frame
        const int b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * zb);
        frame_finalize<MODE == ADJ_CG_INIT ? FIN_RR0 : FIN_ALPHA>(sum, t, b, bpf, cg);
    }
}

// e' = step * e for every ray (input of the gather for a plain A^T).
__global__ void planes_step_weight_kernel(const float4* __restrict__ col, const float* __restrict__ e,
                                   float* __restrict__ out, ProjDims d) {
    const int iu = blockIdx.x * 32 + threadIdx.x;
    const int iv = blockIdx.y * 4 + threadIdx.y;
    const int g = blockIdx.z;
    if (iu >= d.nu || iv >= d.nv) return;
    const ColParams c = load_col(col, (size_t)g * d.nu + iu);
    const RayZ rz = ray_z(c, det_v(iv, d), d.cz);
    const size_t ray = ((size_t)g * d.nv + iv) * d.nu + iu;
    out[ray] = rz.step * e[ray];
}

// ------------------------------------------------------------------ CG vectors

// z += alpha p; r -= alpha q; beta = r.r / rr  (grid: blocks_per_frame x nt).
// Each thread adds the squares of runs of 8 of its elements in FP32 before its
// FP64 sum (FP64 arithmetic is a small fraction of the FP32 rate on this GPU);
// the order of every addition is fixed.
__global__ void planes_cg_update_kernel(float* __restrict__ z, float* __restrict__ r,
                                        const float* __restrict__ p, const float* __restrict__ q,
                                        const double* __restrict__ alpha, CgScalars cg,
                                        size_t fs) {
    const int t = blockIdx.y;
    const float a = (float)alpha[t];
    const size_t off = (size_t)t * fs;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    double dot = 0.0;
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    while (i < fs) {
        float run = 0.0f;
        for (int k = 0; k < 8 && i < fs; ++k, i += stride) {
            z[off + i] = __fmaf_rn(a, p[off + i], z[off + i]);
            const float rn = __fmaf_rn(-a, q[off + i], r[off + i]);
            r[off + i] = rn;
            run = __fmaf_rn(rn, rn, run);
        }
        dot += (double)run;
    }
    const double s = block_sum_f64(dot);
    frame_finalize<FIN_BETA>(s, t, blockIdx.x, gridDim.x, cg);
}

// ------------------------------------------------------------------ grouped ICD (projector.cu states the method)

constexpr int ICD_SINO_BLOCKS = 256;   // blocks per frame of the sinogram passes
constexpr int ICD_ZB = 8;              // group voxels per z-run of the group gather (16 slices)

// Adds, for the rays of one view whose major axis is XMAJ, the gather terms of
// the voxels (ix, iy, base + ZS*j), j < ZB, into acc[j]: w_a w_z e' (SQ false)
// or w_a^2 w_z^2 e' (SQ true, with e' = step^2 Lambda: the diagonal of
// A^T Lambda A).  Candidate columns, the a weight and the affine z crossing per
// row are formed exactly as in gather_runs.
template <bool XMAJ, int ZB, int ZS, bool SQ>
__device__ __forceinline__ void gather_icd(const float4* __restrict__ col, const float* __restrict__ e, int g,
                                           int ix, int iy, int base, float cs, float sn, const ProjDims& d,
                                           float (*acc)[128], int tid) {
    const int kpl = XMAJ ? ix : iy;
    const int ia = XMAJ ? iy : ix;
    const float cmaj = XMAJ ? d.cx : d.cy;
    const float xc = (ix - d.cx) * d.vox, yc = (iy - d.cy) * d.vox;
    float u1, u2;
    if (XMAJ) {
        u1 = u_pixel(xc, yc - d.vox, cs, sn, d);
        u2 = u_pixel(xc, yc + d.vox, cs, sn, d);
    } else {
        u1 = u_pixel(xc - d.vox, yc, cs, sn, d);
        u2 = u_pixel(xc + d.vox, yc, cs, sn, d);
    }
    const int iu_lo = max(0, (int)floorf(fminf(u1, u2)) - 1);
    const int iu_hi = min(d.nu - 1, (int)ceilf(fmaxf(u1, u2)) + 1);
    const float tk = __fsub_rn((float)kpl, cmaj);
    const float inv_dv = 1.0f / d.dv;
    const int zlast = base + ZS * (ZB - 1);
    for (int iu = iu_lo; iu <= iu_hi; ++iu) {
        const ColParams c = load_col(col, (size_t)g * d.nu + iu);
        if ((c.xmajor != 0.0f) != XMAJ) continue;
        const float fa = __fmaf_rn(tk, c.ba, c.fa_mid);
        const float a0f = floorf(fa);
        const int a0 = (int)a0f;
        if (ia != a0 && ia != a0 + 1) continue;
        const float wa1 = __fsub_rn(fa, a0f);
        const float wa = (ia == a0) ? __fsub_rn(1.0f, wa1) : wa1;
        const float wav = SQ ? __fmul_rn(wa, wa) : wa;
        const float rgz = __fdividef(1.0f, c.c1 + tk * c.inv_dmaj);
        const float va = (base - 1 - d.cz) * rgz * inv_dv + d.cv;
        const float vb = (zlast + 1 - d.cz) * rgz * inv_dv + d.cv;
        const int iv_lo = max(0, (int)floorf(va) - 1);
        const int iv_hi = min(d.nv - 1, (int)ceilf(vb) + 1);
        const float* erow = e + ((size_t)g * d.nv) * d.nu + iu;
        const RayZ rzb = ray_z(c, det_v(0, d), d.cz);
        const float fzb = __fmaf_rn(tk, rzb.bz, rzb.fz_mid);
        const float dfz = d.dv * __fmaf_rn(tk, c.inv_dmaj, c.c1);
        for (int iv = iv_lo; iv <= iv_hi; ++iv) {
            const float fz = __fmaf_rn((float)iv, dfz, fzb);
            const float z0f = floorf(fz);
            const int z0 = (int)z0f;
            if (z0 + 1 < base || z0 > zlast) continue;
            const float ev = __fmul_rn(wav, __ldg(erow + (size_t)iv * d.nu));
            const float wz1 = __fsub_rn(fz, z0f);
            const float w1 = SQ ? __fmul_rn(wz1, wz1) : wz1;
            const float w0 = SQ ? __fmul_rn(__fsub_rn(1.0f, wz1), __fsub_rn(1.0f, wz1)) : 0.0f;
            const float c1 = __fmul_rn(w1, ev);
            const float c0 = SQ ? __fmul_rn(w0, ev) : __fsub_rn(ev, c1);
            const int o0 = z0 - base, o1 = z0 + 1 - base;
            if (o0 >= 0 && o0 % ZS == 0 && o0 / ZS < ZB) acc[o0 / ZS][tid] = __fadd_rn(acc[o0 / ZS][tid], c0);
            if (o1 >= 0 && o1 % ZS == 0 && o1 / ZS < ZB) acc[o1 / ZS][tid] = __fadd_rn(acc[o1 / ZS][tid], c1);
        }
    }
}

// theta2 = (A^T Lambda A)_ss + 1/sigma^2 for every voxel: the squared-weight
// gather of e2 = step^2 Lambda.  Grid and runs as joseph_adj_kernel.
template <int ZB>
__global__ void __launch_bounds__(128) planes_icd_theta2_kernel(const float4* __restrict__ col,
                                                         const float2* __restrict__ trig,
                                                         const int* __restrict__ vflag,
                                                         const float* __restrict__ e2, float* __restrict__ theta2,
                                                         float inv_s2, ProjDims d) {
    __shared__ float acc[ZB][128];
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int ix = blockIdx.x * 32 + threadIdx.x;
    const int iy = blockIdx.y * 4 + threadIdx.y;
    const int nzb = (d.nz + ZB - 1) / ZB;
    const int zb = blockIdx.z % nzb, t = blockIdx.z / nzb;
    const int base = zb * ZB;
    const bool inside = ix < d.nx && iy < d.ny;
#pragma unroll
    for (int k = 0; k < ZB; ++k) acc[k][tid] = 0.0f;
    if (inside) {
        for (int j = 0; j < d.views; ++j) {
            const int g = t * d.views + j;
            const float2 cs = __ldg(trig + g);
            const int fl = __ldg(vflag + g);
            if (fl & 1) gather_icd<true, ZB, 1, true>(col, e2, g, ix, iy, base, cs.x, cs.y, d, acc, tid);
            if (fl & 2) gather_icd<false, ZB, 1, true>(col, e2, g, ix, iy, base, cs.x, cs.y, d, acc, tid);
        }
        for (int k = 0; k < ZB && base + k < d.nz; ++k)
            theta2[(((size_t)t * d.nz + base + k) * d.ny + iy) * d.nx + ix] = acc[k][tid] + inv_s2;
    }
}

// The group step's gather: for every voxel s of the group, delta_s =
// -theta1_s/theta2_s (written to dlt), and per-block partial sums of
// theta1.delta and delta.delta (FP64, fixed order).  A thread owns one group
// column (ix, iy) and a run of ZB group voxels along z (stride 2).
template <int ZB>
__global__ void __launch_bounds__(128) planes_icd_group_kernel(const float4* __restrict__ col,
                                                        const float2* __restrict__ trig,
                                                        const int* __restrict__ vflag, const float* __restrict__ e,
                                                        const float* __restrict__ z, const float* __restrict__ v,
                                                        const float* __restrict__ theta2, float* __restrict__ dlt,
                                                        double* __restrict__ gpart, float inv_s2, IcdGroup G,
                                                        ProjDims d) {
    __shared__ float acc[ZB][128];
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int jx = blockIdx.x * 32 + threadIdx.x, jy = blockIdx.y * 4 + threadIdx.y;
    const int ix = 2 * jx + G.px, iy = 2 * jy + G.py;
    const int nzb = (G.gz + ZB - 1) / ZB, zb = blockIdx.z % nzb, t = blockIdx.z / nzb;
    const int base = G.pz + 2 * ZB * zb;
    const bool inside = jx < G.gx && jy < G.gy;
#pragma unroll
    for (int k = 0; k < ZB; ++k) acc[k][tid] = 0.0f;
    if (inside) {
        for (int j = 0; j < d.views; ++j) {
            const int g = t * d.views + j;
            const float2 cs = __ldg(trig + g);
            const int fl = __ldg(vflag + g);
            if (fl & 1) gather_icd<true, ZB, 2, false>(col, e, g, ix, iy, base, cs.x, cs.y, d, acc, tid);
            if (fl & 2) gather_icd<false, ZB, 2, false>(col, e, g, ix, iy, base, cs.x, cs.y, d, acc, tid);
        }
    }
    double gd = 0.0, dd = 0.0;
    for (int k = 0; k < ZB; ++k) {
        const int iz = base + 2 * k;
        if (!inside || iz >= d.nz) break;
        const size_t i = (((size_t)t * d.nz + iz) * d.ny + iy) * d.nx + ix;
        const float th1 = __fmaf_rn(__fsub_rn(z[i], v[i]), inv_s2, -acc[k][tid]);
        const float del = -__fdiv_rn(th1, theta2[i]);
        dlt[i] = del;
        gd += (double)th1 * (double)del;
        dd += (double)del * (double)del;
    }
    const double sg = block_sum_f64(gd);
    const double sd = block_sum_f64(dd);
    if (tid == 0) {
        const int bpf = gridDim.x * gridDim.y * nzb;
        const int b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * zb);
        gpart[2 * ((size_t)t * bpf + b)] = sg;
        gpart[2 * ((size_t)t * bpf + b) + 1] = sd;
    }
}

// Sinogram passes of a group step, per frame (grid ICD_SINO_BLOCKS x nt):
//   PASS 0: the sum of Lambda (A delta)^2, and the line search's alpha (icd_alpha)
//   PASS 1: e' -= alpha_t step Lambda (A delta)
// ad = A delta (plain forward), lam = Lambda, e' the step-weighted residual.
template <int PASS>
__global__ void __launch_bounds__(256) planes_icd_sino_kernel(const float4* __restrict__ col,
                                                       const float* __restrict__ ad, const float* __restrict__ lam,
                                                       float* __restrict__ e, IcdSums S, ProjDims d) {
    const int t = blockIdx.y;
    const size_t per_view = (size_t)d.nu * d.nv, mt = per_view * d.views;
    const size_t off = (size_t)t * mt;
    const float a = PASS == 1 ? (float)S.alpha[t] : 0.0f;
    double s = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < mt; i += (size_t)gridDim.x * blockDim.x) {
        const float val = ad[off + i];
        const float l = lam[off + i];
        if (PASS == 0) {
            s += (double)l * (double)val * (double)val;
        } else {
            const int j = (int)(i / per_view);
            const int iv = (int)((i % per_view) / d.nu), iu = (int)(i % d.nu);
            const ColParams c = load_col(col, ((size_t)t * d.views + j) * d.nu + iu);
            const float step = ray_z(c, det_v(iv, d), d.cz).step;
            e[off + i] = __fmaf_rn(-a, __fmul_rn(step, __fmul_rn(l, val)), e[off + i]);
        }
    }
    if (PASS == 0) {
        const double sum = block_sum_f64(s);
        icd_alpha(sum, t, blockIdx.x, gridDim.x, S);
    }
}

// z_s += alpha_t delta_s and delta_s = 0 for the voxels of the group.
__global__ void planes_icd_update_kernel(float* __restrict__ z, float* __restrict__ dlt, const double* __restrict__ alpha,
                                  IcdGroup G, ProjDims d) {
    const size_t per_frame = (size_t)G.gx * G.gy * G.gz;
    const size_t total = per_frame * d.nt;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(i / per_frame);
        size_t r = i % per_frame;
        const int jz = (int)(r / ((size_t)G.gx * G.gy));
        r %= (size_t)G.gx * G.gy;
        const int jy = (int)(r / G.gx), jx = (int)(r % G.gx);
        const size_t k = (((size_t)t * d.nz + 2 * jz + G.pz) * d.ny + 2 * jy + G.py) * d.nx + 2 * jx + G.px;
        z[k] = __fmaf_rn((float)alpha[t], dlt[k], z[k]);
        dlt[k] = 0.0f;
    }
}

// e2 = step^2 Lambda for every ray (input of the theta2 gather).
__global__ void planes_icd_step2_kernel(const float4* __restrict__ col, const float* __restrict__ lam,
                                 float* __restrict__ out, ProjDims d) {
    const int iu = blockIdx.x * 32 + threadIdx.x;
    const int iv = blockIdx.y * 4 + threadIdx.y;
    const int g = blockIdx.z;
    if (iu >= d.nu || iv >= d.nv) return;
    const ColParams c = load_col(col, (size_t)g * d.nu + iu);
    const float step = ray_z(c, det_v(iv, d), d.cz).step;
    const size_t ray = ((size_t)g * d.nv + iv) * d.nu + iu;
    out[ray] = __fmul_rn(__fmul_rn(step, step), lam[ray]);
}

// ====================================================================== launches

static msf_status launch_pairs(msf_projector* p, const float* in, cudaStream_t st) {
    const msf_vol& v = p->vol;
    dim3 grid((v.nx + 31) / 32, (v.ny + 31) / 32, v.nz * v.nt);
    MSF_PROF("transpose", st);
    pair_kernel<false><<<grid, dim3(32, 8), 0, st>>>(in, p->d_px, p->d_py, nullptr, nullptr, nullptr, v.nx, v.ny, v.nz);
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

// A of the volume whose pairs the plan holds: fwd_bx columns x PLANES_R * fwd_by rows per block, one z per view.
template <int MODE, bool PAR = false>
static msf_status launch_fwd_pairs(msf_projector* p, float* out, const float* lam, const float* meas, cudaStream_t st,
                                   int kpx = 0, int kpy = 0) {
    const ProjDims& d = p->dims;
    const dim3 block(p->fwd_bx, p->fwd_by);
    const unsigned rows = block.y * PLANES_R;
    const dim3 grid((d.nu + block.x - 1) / block.x, (d.nv + rows - 1) / rows, d.nt * d.views);
    MSF_PROF("joseph_fwd", st);
    planes_fwd_kernel<MODE, PAR><<<grid, block, 0, st>>>(p->d_px, p->d_py, p->d_col, out, lam, meas, d, kpx, kpy);
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

static int nzb_of(const ProjDims& d, int zb) { return (d.nz + zb - 1) / zb; }
static dim3 adj_grid(const ProjDims& d, int zb) { return dim3((d.nx + 31) / 32, (d.ny + 3) / 4, nzb_of(d, zb) * d.nt); }

template <int MODE>
static msf_status launch_adj(msf_projector* p, const float* e, float* out, const float* a1, const float* a2, float* out2,
                             const CgScalars& cg, float inv_s2, cudaStream_t st) {
    const ProjDims& d = p->dims;
    MSF_PROF("joseph_adj", st);
#define MSF_ADJ_CASE(ZB)                                                                                            \
    case ZB:                                                                                                        \
        planes_adj_kernel<MODE, ZB><<<adj_grid(d, ZB), dim3(32, 4), 0, st>>>(p->d_col, p->d_trig, p->d_vflag, e, out, a1, \
                                                                             a2, out2, cg, inv_s2, d);              \
        break;
    switch (p->adj_zb) {
        MSF_ADJ_CASE(8)
        MSF_ADJ_CASE(16)
        MSF_ADJ_CASE(32)
        MSF_ADJ_CASE(64)
    }
#undef MSF_ADJ_CASE
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

// the launch grids' z: slices, views and runs of 8 slices of all frames
bool planes_fit(const ProjDims& d) {
    const long long z = 65535;
    return (long long)d.nz * d.nt <= z && (long long)d.views * d.nt <= z;
}

msf_status planes_project(msf_projector* p, const float* x, float* y, cudaStream_t st) {
    MSF_TRY(launch_pairs(p, x, st));
    return launch_fwd_pairs<FWD_PLAIN>(p, y, nullptr, nullptr, st);
}

msf_status planes_project_pairs(msf_projector* p, float* y, cudaStream_t st) {
    return launch_fwd_pairs<FWD_PLAIN>(p, y, nullptr, nullptr, st);
}

msf_status planes_gather(msf_projector* p, const float* e, float* x, cudaStream_t st) {
    return launch_adj<ADJ_PLAIN>(p, e, x, nullptr, nullptr, nullptr, CgScalars{}, 0.0f, st);
}

int planes_adj_blocks(const ProjDims& d, int zb) {
    const dim3 g = adj_grid(d, zb);
    return g.x * g.y * nzb_of(d, zb);
}

msf_status planes_backproject(msf_projector* p, const float* y, float* x, cudaStream_t st) {
    const ProjDims& d = p->dims;
    {
        MSF_PROF("step_weight", st);
        planes_step_weight_kernel<<<dim3((d.nu + 31) / 32, (d.nv + 3) / 4, d.nt * d.views), dim3(32, 4), 0, st>>>(
            p->d_col, y, p->d_sw, d);
        MSF_LAUNCH_CHECK();
    }
    return planes_gather(p, p->d_sw, x, st);
}

// ====================================================================== data agents

msf_status planes_dataprox_alloc(msf_dataprox* d, size_t sino, size_t ipart, size_t spart) {
    const msf_projector* p = d->p;
    const msf_vol& v = p->vol;
    const size_t n = vol_size(v), ns = std::max(sino, sino_size(p)), nt = v.nt;
    d->parts_upd = 512;
    const int parts = std::max(planes_adj_blocks(p->dims, 8), d->parts_upd);   // the largest block count of any z-run
    const size_t parts_icd = (size_t)((par_count(v.nx, 0) + 31) / 32) * ((par_count(v.ny, 0) + 3) / 4) *
                             ((par_count(v.nz, 0) + ICD_ZB - 1) / ICD_ZB);     // parity 0 along every axis: the largest group
    if (cudaMalloc(&d->d_r, 4 * n * 4) != cudaSuccess || cudaMalloc(&d->d_rows, ns * 4) != cudaSuccess ||
        cudaMalloc(&d->d_rows2, ns * 4) != cudaSuccess ||
        cudaMalloc(&d->d_ipart, std::max(ipart, nt * parts_icd * 2) * 8) != cudaSuccess ||
        cudaMalloc(&d->d_spart, std::max(spart, nt * ICD_SINO_BLOCKS) * 8) != cudaSuccess ||
        cudaMalloc(&d->d_partial, nt * parts * 8) != cudaSuccess)
        return MSF_ERR_NOMEM;
    d->d_p = d->d_r + n;
    d->d_p2 = d->d_p + n;
    d->d_q = d->d_p2 + n;
    return MSF_OK;
}

msf_status planes_prox_cg(msf_dataprox* dp, const float* y, const float* lambda, const float* v, float* x, float inv_s2,
                          int n_cg, cudaStream_t st) {
    msf_projector* p = dp->p;
    const msf_vol& vol = p->vol;
    const int nt = vol.nt;
    const CgScalars ca{dp->d_partial, dp->d_rr, dp->d_alpha, dp->d_status, dp->d_count};
    const CgScalars cb{dp->d_partial, dp->d_rr, dp->d_beta, dp->d_status, dp->d_count};
    // r = A^T Lambda (y - A z) + (v - z)/sigma^2 ; p = r ; rr = r.r
    MSF_TRY(launch_pairs(p, x, st));
    MSF_TRY(launch_fwd_pairs<FWD_RESIDUAL>(p, dp->d_rows, lambda, y, st));
    MSF_TRY(launch_adj<ADJ_CG_INIT>(p, dp->d_rows, dp->d_r, v, x, dp->d_p, ca, inv_s2, st));
    // the direction p alternates between two buffers: the fused update reads
    // p at slices z and z + 1 while writing the new p
    float* pc = dp->d_p;
    for (int it = 0; it < n_cg; ++it) {
        // z-paired copies of p for the forward (fused with p = r + beta p after the first step)
        if (it == 0) {
            MSF_TRY(launch_pairs(p, pc, st));
        } else {
            float* pn = pc == dp->d_p ? dp->d_p2 : dp->d_p;
            MSF_PROF("transpose_pupdate", st);
            pair_kernel<true><<<dim3((vol.nx + 31) / 32, (vol.ny + 31) / 32, vol.nz * nt), dim3(32, 8), 0, st>>>(
                pc, p->d_px, p->d_py, dp->d_r, pn, dp->d_beta, vol.nx, vol.ny, vol.nz);
            MSF_LAUNCH_CHECK();
            pc = pn;
        }
        // s = Lambda A p ; q = A^T s + p/sigma^2 ; alpha = rr / p.q
        MSF_TRY(launch_fwd_pairs<FWD_LAMBDA>(p, dp->d_rows, lambda, nullptr, st));
        MSF_TRY(launch_adj<ADJ_CG_Q>(p, dp->d_rows, dp->d_q, pc, nullptr, nullptr, ca, inv_s2, st));
        // z += alpha p ; r -= alpha q ; beta = r.r / rr
        MSF_PROF("cg_update", st);
        planes_cg_update_kernel<<<dim3(dp->parts_upd, nt), 256, 0, st>>>(x, dp->d_r, pc, dp->d_q, dp->d_alpha, cb,
                                                                         frame_size(vol));
        MSF_LAUNCH_CHECK();
    }
    return MSF_OK;
}

msf_status planes_prox_icd(msf_dataprox* dp, const float* y, const float* lambda, const float* v, float* x, double sigma,
                           int n_sweeps, cudaStream_t st) {
    msf_projector* p = dp->p;
    const ProjDims& d = p->dims;
    const msf_vol& vol = p->vol;
    const int nt = vol.nt;
    const float inv_s2 = (float)(1.0 / (sigma * sigma));
    float *e = dp->d_rows, *ad = dp->d_rows2, *theta2 = dp->d_q, *dlt = dp->d_p;
    // e' = step Lambda (y - A z)
    MSF_TRY(launch_pairs(p, x, st));
    MSF_TRY(launch_fwd_pairs<FWD_RESIDUAL>(p, e, lambda, y, st));
    {   // theta2 = (A^T Lambda A)_ss + 1/sigma^2
        MSF_PROF("icd_weights", st);
        planes_icd_step2_kernel<<<dim3((d.nu + 31) / 32, (d.nv + 3) / 4, nt * d.views), dim3(32, 4), 0, st>>>(
            p->d_col, lambda, ad, d);
        MSF_LAUNCH_CHECK();
    }
    {
        MSF_PROF("icd_theta2", st);
        planes_icd_theta2_kernel<16><<<adj_grid(d, 16), dim3(32, 4), 0, st>>>(p->d_col, p->d_trig, p->d_vflag, ad, theta2,
                                                                              inv_s2, d);
        MSF_LAUNCH_CHECK();
    }
    MSF_TRY_CUDA(cudaMemsetAsync(dlt, 0, vol_size(vol) * sizeof(float), st));
    IcdSums S{dp->d_ipart, dp->d_spart, 0, dp->d_alpha, 1.0 / (sigma * sigma), dp->d_status, dp->d_count};
    for (int sw = 0; sw < n_sweeps; ++sw) {
        for (int grp = 0; grp < 8; ++grp) {
            IcdGroup G;
            G.px = grp & 1; G.py = (grp >> 1) & 1; G.pz = grp >> 2;
            G.gx = par_count(vol.nx, G.px); G.gy = par_count(vol.ny, G.py); G.gz = par_count(vol.nz, G.pz);
            if (G.gx == 0 || G.gy == 0 || G.gz == 0) continue;
            const int nzb = (G.gz + ICD_ZB - 1) / ICD_ZB;
            const dim3 grid((G.gx + 31) / 32, (G.gy + 3) / 4, nzb * nt);
            S.gblocks = grid.x * grid.y * nzb;
            {
                MSF_PROF("icd_group", st);
                planes_icd_group_kernel<ICD_ZB><<<grid, dim3(32, 4), 0, st>>>(p->d_col, p->d_trig, p->d_vflag, e, x, v,
                                                                              theta2, dlt, dp->d_ipart, inv_s2, G, d);
                MSF_LAUNCH_CHECK();
            }
            // A delta: delta is zero outside the group (the update clears it)
            MSF_TRY(launch_pairs(p, dlt, st));
            MSF_TRY((launch_fwd_pairs<FWD_PLAIN, true>(p, ad, nullptr, nullptr, st, G.px, G.py)));
            {
                MSF_PROF("icd_sino", st);
                planes_icd_sino_kernel<0><<<dim3(ICD_SINO_BLOCKS, nt), 256, 0, st>>>(p->d_col, ad, lambda, e, S, d);
                MSF_LAUNCH_CHECK();
            }
            {
                MSF_PROF("icd_update", st);
                planes_icd_update_kernel<<<152 * 4, 256, 0, st>>>(x, dlt, dp->d_alpha, G, d);
                MSF_LAUNCH_CHECK();
            }
            {
                MSF_PROF("icd_sino", st);
                planes_icd_sino_kernel<1><<<dim3(ICD_SINO_BLOCKS, nt), 256, 0, st>>>(p->d_col, ad, lambda, e, S, d);
                MSF_LAUNCH_CHECK();
            }
        }
    }
    return MSF_OK;
}

}  // namespace msf
