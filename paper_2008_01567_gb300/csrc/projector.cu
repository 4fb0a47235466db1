// Cone-beam Joseph projector pair and the CG data proximal map.
//
// A_n (Sec. II, Eq. (2)) is modelled as a Joseph ray-driven projector on a
// circular orbit with a flat detector (the paper defers the model to its
// cone-beam reference; the geometry is documented in msf.h).  The adjoint is a
// voxel-driven gather: each voxel enumerates the rays whose bilinear footprint
// touches it and recomputes the forward's interpolation coordinates with the
// same FP32 operations (the z crossing to within a few 1e-5 voxel): A^T is the
// transpose of the FP32 A up to rounding, without atomics.
//
// Per (view, detector column) constants are computed once in FP64 and stored
// in FP32.  A ray's direction has d_x, d_y fixed by its column and d_z = v, so
// the in-plane constants are per column and the z constants are v times
// per-column factors.  Along the major axis the crossing point at plane k is
//     f_a(k) = fa_mid + (k - c_maj) * ba          (minor in-plane axis)
//     f_z(k) = (c_z + v*c1) + (k - c_maj) * (v*inv_dmaj)
// in fractional voxel indices, and the chord per plane is
//     step = sqrt(|d_xy|^2 + v^2) * voxel/|d_maj|.
//
// The kernels here take a warp's lanes along detector rows and along z, on volumes in
// lines along z; thin detectors and volumes take those of projector_planes.cu
// (choose_routes).
#include <math.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "projector.cuh"

namespace msf {

// ------------------------------------------------------------------ FP64 table

// One thread per (frame-view g, column iu).  Writes the column constants and
// flags geometry the model does not cover: a plane crossing outside the
// source-detector segment (0 < lambda < 1) on the first or last plane.
__global__ void column_table_kernel(const double* __restrict__ angles, float4* __restrict__ col,
                                    int* __restrict__ vflag, int* __restrict__ bad, ProjDims d,
                                    double vox, double du, double dso, double dsd) {
    const int iu = blockIdx.x * blockDim.x + threadIdx.x;
    const int g = blockIdx.y;
    if (iu >= d.nu) return;
    const double th = angles[g];
    const double c = cos(th), s = sin(th);
    const double u = (iu - 0.5 * (d.nu - 1)) * du;
    const double sx = dso * c, sy = dso * s;
    const double px = -(dsd - dso) * c - u * s;
    const double py = -(dsd - dso) * s + u * c;
    const double dx = px - sx, dy = py - sy;
    const bool xmaj = fabs(dx) >= fabs(dy);
    const double dmaj = xmaj ? dx : dy, smaj = xmaj ? sx : sy;
    const double da = xmaj ? dy : dx, sa = xmaj ? sy : sx;
    const int nmaj = xmaj ? d.nx : d.ny, na = xmaj ? d.ny : d.nx;
    const double lam0 = -smaj / dmaj;
    float4 a, b;
    a.x = (float)((sa + lam0 * da) / vox + 0.5 * (na - 1));
    a.y = (float)(da / dmaj);
    a.z = (float)(lam0 / vox);
    a.w = (float)(1.0 / dmaj);
    b.x = (float)(dx * dx + dy * dy);
    b.y = (float)(vox / fabs(dmaj));
    b.z = xmaj ? 1.0f : 0.0f;
    b.w = 0.0f;
    const size_t idx = (size_t)g * d.nu + iu;
    col[2 * idx] = a;
    col[2 * idx + 1] = b;
    atomicOr(vflag + g, xmaj ? 1 : 2);   // which major axes occur in this view
    const double lfirst = lam0 + (0 - 0.5 * (nmaj - 1)) * vox / dmaj;
    const double llast = lam0 + (nmaj - 1 - 0.5 * (nmaj - 1)) * vox / dmaj;
    if (!(fmin(lfirst, llast) > 0.0 && fmax(lfirst, llast) < 1.0)) atomicExch(bad, 1);
    (void)na;
}

// ------------------------------------------------------------------ z-contiguous copies

// The forward reads a frame as lines of voxels along z: line (y, x) of frame t
// starts at VZ_FRONT + ((t*ny + y)*nx + x) * nzp.  The elements between the lines
// (two or more, shared by a line's end and the next one's start) and the VZ_FRONT
// before the first are zeros that nothing writes (the buffers are cleared when they
// are allocated), so that a tap outside the volume in z reads 0 without a check.
// (With margins of each line's own a volume of one slice took 32 bytes per voxel,
// now 16; lines start on 16 bytes either way.)
constexpr int VZ_FRONT = 4;
__host__ __device__ __forceinline__ int vz_pitch(int nz) { return (nz + 2 + 3) & ~3; }

// Transposes between a volume [nt][nz][ny][nx] and its lines, through 64 x 64
// shared tiles of one (t, y) plane: 256-byte pieces on both sides, 16 loads per
// thread in flight.  Bound by HBM.
enum LinesMode { LINES_COPY = 0, LINES_PAIR = 1, LINES_BOTH = 2 };
constexpr int LT = 64;

// LINES_COPY: vz = lines of in.  LINES_PAIR: also vd = lines of v - in; LINES_BOTH:
// also vd = lines of v.  margins: also clears those of vz (a plan that keeps pairs in
// the same place).
template <int MODE>
__global__ void __launch_bounds__(256) lines_kernel(const float* __restrict__ in, float* __restrict__ vz,
                                                    const float* __restrict__ v, float* __restrict__ vd, int nx, int ny,
                                                    int nz, bool margins) {
    __shared__ float tile[LT][LT + 1];
    const int xt = (nx + LT - 1) / LT, ty = blockIdx.x / xt, t = ty / ny, y = ty % ny;
    const int x0 = blockIdx.x % xt * LT, z0 = blockIdx.y * LT;
    const int nzp = vz_pitch(nz);
    const int lo = threadIdx.x % LT, hi = threadIdx.x / LT;
    constexpr bool TWO = MODE != LINES_COPY;
    float keep[TWO ? LT / 4 : 1];
#pragma unroll
    for (int k = 0; k < LT / 4; ++k) {
        const int x = x0 + lo, z = z0 + 4 * k + hi;
        const bool ok = x < nx && z < nz;
        const size_t i = (((size_t)t * nz + z) * ny + y) * nx + x;
        const float a = ok ? in[i] : 0.0f;
        if (TWO) keep[k] = !ok ? 0.0f : MODE == LINES_PAIR ? __fsub_rn(v[i], a) : v[i];
        tile[4 * k + hi][lo] = a;
    }
#pragma unroll
    for (int pass = 0; pass < (TWO ? 2 : 1); ++pass) {
        float* out = pass ? vd : vz;
        if (pass) {
            __syncthreads();
#pragma unroll
            for (int k = 0; k < LT / 4; ++k) tile[4 * k + hi][lo] = keep[TWO ? k : 0];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < LT / 4; ++k) {
            const int x = x0 + 4 * k + hi, z = z0 + lo;
            if (x < nx && z < nz) out[(((size_t)t * ny + y) * nx + x) * nzp + VZ_FRONT + z] = tile[lo][4 * k + hi];
        }
    }
    if (margins && blockIdx.y == 0) {
        const int m = nzp - nz;
        for (int i = threadIdx.x; i < LT * m && x0 + i / m < nx; i += blockDim.x)
            vz[(((size_t)t * ny + y) * nx + x0 + i / m) * nzp + VZ_FRONT + nz + i % m] = 0.0f;
        if (blockIdx.x == 0 && threadIdx.x < VZ_FRONT) vz[threadIdx.x] = 0.0f;
    }
}

// x[nt][nz][ny][nx] = z (+ alpha_t p), z and p as lines (ADD: the last CG step, whose new
// residual r - alpha_t q has no reader: squared and added by eights, as cg_residual_kernel
// would, it raises the status flag if that is not finite).
template <bool ADD>
__global__ void __launch_bounds__(256) volume_kernel(const float* __restrict__ vz, const float* __restrict__ p,
                                                     const float* __restrict__ r, const float* __restrict__ q,
                                                     const double* __restrict__ alpha, float* __restrict__ out,
                                                     int* __restrict__ status, int nx, int ny, int nz) {
    __shared__ float tile[LT][LT + 1];
    const int xt = (nx + LT - 1) / LT, ty = blockIdx.x / xt, t = ty / ny, y = ty % ny;
    const int x0 = blockIdx.x % xt * LT, z0 = blockIdx.y * LT;
    const int nzp = vz_pitch(nz);
    const int lo = threadIdx.x % LT, hi = threadIdx.x / LT;
    const float a = ADD ? (float)alpha[t] : 0.0f;
    bool ok = true;
#pragma unroll
    for (int k0 = 0; k0 < LT / 4; k0 += 8) {   // eight voxels' loads before their sums
        float zv[8], pv[8], rv[8], qv[8], run = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x = x0 + 4 * (k0 + k) + hi, z = z0 + lo;
            const bool in = x < nx && z < nz;
            const size_t i = (((size_t)t * ny + y) * nx + x) * nzp + VZ_FRONT + z;
            zv[k] = in ? vz[i] : 0.0f;
            pv[k] = ADD && in ? p[i] : 0.0f;
            rv[k] = ADD && in ? r[i] : 0.0f;
            qv[k] = ADD && in ? q[i] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            tile[lo][4 * (k0 + k) + hi] = ADD ? __fmaf_rn(a, pv[k], zv[k]) : zv[k];
            const float rn = __fmaf_rn(-a, qv[k], rv[k]);
            run = __fmaf_rn(rn, rn, run);
        }
        ok = ok && isfinite(run);
    }
    if (ADD && !ok) atomicExch(status, (int)MSF_ERR_NUMERIC);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < LT / 4; ++k) {
        const int x = x0 + lo, z = z0 + 4 * k + hi;
        if (x < nx && z < nz) out[(((size_t)t * nz + z) * ny + y) * nx + x] = tile[4 * k + hi][lo];
    }
}

// ------------------------------------------------------------------ forward

// Row sets (32 detector rows each) of one warp.  Five sets share a plane's
// in-plane arithmetic among the most rays (160 rows: 0.67 ms in one chunk of
// five, 0.86 in two of three); up to four sets two planes are unrolled under a
// limit of three blocks per SM, which keeps their loads in flight (384 rows:
// 2.43 ms in chunks of four, 2.76 without the limit, 2.69 in chunks of six,
// whose slab of z-slices also leaves L2).
constexpr int FWD_MAX_R = 5;

// The step-weighted sinogram e' as the gather reads it: lines of detector rows,
// row iv of (view g, column iu) at SINO_FRONT + (g*nu + iu) * sino_pitch + iv.
// The elements between the lines (SINO_FRONT or more, shared) and before the first
// are zeros that nothing writes: rows a voxel's window reaches beyond the detector
// read 0.
constexpr int SINO_FRONT = 4;
__host__ __device__ __forceinline__ int sino_pitch(int nv) { return (nv + SINO_FRONT + 3) & ~3; }

// 2^23 + 2^22: adding it in round-down mode leaves floor(f) in the low mantissa
// bits for |f| < 2^22, so the floor and its integer cost two additions instead
// of two conversions.
constexpr float FLOOR_MAGIC = 12582912.0f;
constexpr int FLOOR_MAGIC_BITS = 0x4B400000;

// A warp takes one detector column and R sets of 32 consecutive rows (lane =
// row in a set); a block takes blockDim.y neighbouring columns.  All rays of a
// column lie in one vertical plane: on voxel plane k of the major axis they
// share the in-plane crossing f_a, so the warp forms it once for its R sets and
// reads two z-lines (a0 and a0 + 1), along which the lanes step by the row
// spacing.  Bound by L1 wavefronts: a crossing is four 4-byte loads, and a load
// of 32 lanes (a span of 32 row spacings, on any alignment) takes 1.86.  With
// lanes along u and 8-byte loads of z-paired copies (16 bytes of copies per
// voxel) it took 8.8 for each of two loads: 30.1 -> 16.6 ms at 384^3 x 16, 512 x
// 384 detector, 24 views (740 G crossings/s); 0.90 -> 0.62 ms at 128^3 x 8, 192 x
// 160, 32 views; 25 -> 10 us at 24^3 x 4, 32 x 32, 12 views.  Pairs of sets
// share instructions (f32x2), since at 30 instructions per crossing the issue
// slots bound it as much (2.43 against 2.59 ms at 384^3 x 2).
// The interpolation is v00 + w_a (v01 - v00) along a, then the same along z,
// summed over increasing planes.  A line outside the volume in a is the zero
// line; f_z is clamped to [-2, nz], where both taps are zeros of the line's
// margins, so a lane outside the volume adds exactly zero.
//   FWD_PLAIN:    out = A x
//   FWD_LAMBDA:   out = step * Lambda * (A x)
//   FWD_RESIDUAL: out = step * Lambda * (meas - A x)
//   FWD_ICD:      out = (step * Lambda) * (A x), and the line search's alpha (icd_alpha)
// (the CG modes write the step-weighted sinogram e' = step * e that the gather
// adjoint consumes; ROWS: as lines of detector rows, sino_pitch).  The sums go
// through shared memory so that the sinogram is read and written in 16-byte
// pieces along u.
// Blocks run over the columns and views of one set of rows before the next:
// the rows of a set cross a slab of z-slices that stays in L2 for all views.
// PAR (the ICD agent's projection of a group step): x is zero outside one
// voxel parity group, so an x-major ray only visits planes x = kpx (mod 2) and
// a y-major ray planes y = kpy (mod 2), and on a visited plane it loads only
// the line of the minor-axis tap with the group's parity (the other is zero);
// the skipped terms are exact zeros, so the result equals the full projection
// bit for bit.
template <int MODE, int R, bool PAR, bool ROWS>
__global__ void __launch_bounds__(256, R == 5 ? 1 : 3) joseph_fwd_kernel(
    const float* __restrict__ vz, const float* __restrict__ zero_line, const float4* __restrict__ col,
    float* __restrict__ out, const float* __restrict__ lam, const float* __restrict__ meas, ProjDims d, int kpx,
    int kpy, IcdSums S) {
    extern __shared__ float fwd_sum[];   // [32 R rows][columns + 1]
    const int lane = threadIdx.x, ncol = blockDim.y;
    const int ublocks = (d.nu + ncol - 1) / ncol;
    const int iu0 = (blockIdx.x % ublocks) * ncol, iu = iu0 + threadIdx.y;
    const int iv0 = blockIdx.y * 32 * R;
    const int t = blockIdx.z, g = t * d.views + blockIdx.x / ublocks;
    if (iu < d.nu) {
        const ColParams c = load_col(col, (size_t)g * d.nu + iu);
        const bool xmaj = c.xmajor != 0.0f;
        const int nmaj = xmaj ? d.nx : d.ny, na = xmaj ? d.ny : d.nx;
        const int nzp = vz_pitch(d.nz);
        // element strides of the major and the minor in-plane axis
        const ptrdiff_t smaj = xmaj ? nzp : (ptrdiff_t)d.nx * nzp, smin = xmaj ? (ptrdiff_t)d.nx * nzp : nzp;
        const float* vol = vz + (size_t)t * d.ny * d.nx * nzp + VZ_FRONT;
        const float* zl = zero_line + VZ_FRONT;
        const float cmaj = xmaj ? d.cx : d.cy;
        const float zmax = (float)d.nz;
        // f_z of the rows, packed by pairs of sets; the last set of an odd R alone
        float f_mid[R], f_b[R];
        // planes where a crossing of the warp can touch the grid (-1 < f < n on
        // both minor axes, one plane of margin)
        int K0 = nmaj, K1 = -1;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const RayZ rz = ray_z(c, det_v(min(iv0 + 32 * r + lane, d.nv - 1), d), d.cz);
            f_mid[r] = rz.fz_mid;
            f_b[r] = rz.bz;
            float lo = 0.0f, hi = (float)(nmaj - 1);
            const float fm[2] = {c.fa_mid, rz.fz_mid}, bb[2] = {c.ba, rz.bz};
            const float top[2] = {(float)na, (float)d.nz};
#pragma unroll
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
                K0 = min(K0, (int)lo);
                K1 = max(K1, (int)hi);
            }
        }
        f32x2 fzm[R / 2 + 1], bz[R / 2 + 1], acc[R / 2 + 1];
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            fzm[r] = pack2(f_mid[2 * r], f_mid[2 * r + 1]);
            bz[r] = pack2(f_b[2 * r], f_b[2 * r + 1]);
            acc[r] = 0;
        }
        const float fzm1 = f_mid[R - 1], bz1 = f_b[R - 1];
        float acc1 = 0.0f;
        K0 = __reduce_min_sync(0xffffffffu, K0);
        K1 = __reduce_max_sync(0xffffffffu, K1);
        const int kp = xmaj ? kpx : kpy, ka = xmaj ? kpy : kpx;
        if (PAR) K0 += (K0 ^ kp) & 1;
        const float* lk = vol + K0 * smaj;   // lines of plane k
        float tk = __fsub_rn((float)K0, cmaj);
#pragma unroll(R == 5 ? 1 : R == 1 ? 4 : 2)
        for (int k = K0; k <= K1; k += PAR ? 2 : 1) {
            const float fa = __fmaf_rn(tk, c.ba, c.fa_mid);
            const float am = __fadd_rd(fa, FLOOR_MAGIC);
            const float wa1 = __fsub_rn(fa, __fsub_rn(am, FLOOR_MAGIC));
            const int ia = __float_as_int(am) - FLOOR_MAGIC_BITS;
            const float* l0 = lk + ia * smin;
            const float* l1 = l0 + smin;
            if ((unsigned)ia >= (unsigned)na) l0 = zl;
            if ((unsigned)(ia + 1) >= (unsigned)na) l1 = zl;
            // PAR: the line of the tap with the group's parity
            const bool first = (ia & 1) == ka;
            // the lines' addresses less the bits of FLOOR_MAGIC, which every index carries
            l0 -= FLOOR_MAGIC_BITS;
            l1 -= FLOOR_MAGIC_BITS;
            const f32x2 tk2 = pack2(tk, tk), wa2 = pack2(wa1, wa1), m2 = pack2(FLOOR_MAGIC, FLOOR_MAGIC);
#pragma unroll
            for (int r = 0; r < R / 2; ++r) {
                float f0, f1;
                unpack2(fma2(tk2, bz[r], fzm[r]), f0, f1);
                const f32x2 fz = pack2(fminf(fmaxf(f0, -2.0f), zmax), fminf(fmaxf(f1, -2.0f), zmax));
                const f32x2 zm = add2_rd(fz, m2);
                const f32x2 wz = sub2(fz, sub2(zm, m2));
                float i0, i1;
                unpack2(zm, i0, i1);
                const int j0 = __float_as_int(i0), j1 = __float_as_int(i1);
                f32x2 v00 = 0, v10 = 0, v01 = 0, v11 = 0;
                if (!PAR || first) {
                    v00 = pack2(__ldg(l0 + j0), __ldg(l0 + j1));
                    v10 = pack2(__ldg(l0 + j0 + 1), __ldg(l0 + j1 + 1));
                }
                if (!PAR || !first) {
                    v01 = pack2(__ldg(l1 + j0), __ldg(l1 + j1));
                    v11 = pack2(__ldg(l1 + j0 + 1), __ldg(l1 + j1 + 1));
                }
                const f32x2 top = fma2(wa2, sub2(v01, v00), v00);
                const f32x2 bot = fma2(wa2, sub2(v11, v10), v10);
                acc[r] = add2(acc[r], fma2(wz, sub2(bot, top), top));
            }
            if (R & 1) {
                const float fz = fminf(fmaxf(__fmaf_rn(tk, bz1, fzm1), -2.0f), zmax);
                const float zm = __fadd_rd(fz, FLOOR_MAGIC);
                const float wz1 = __fsub_rn(fz, __fsub_rn(zm, FLOOR_MAGIC));
                const int j = __float_as_int(zm);
                float v00 = 0.0f, v10 = 0.0f, v01 = 0.0f, v11 = 0.0f;
                if (!PAR || first) {
                    v00 = __ldg(l0 + j);
                    v10 = __ldg(l0 + j + 1);
                }
                if (!PAR || !first) {
                    v01 = __ldg(l1 + j);
                    v11 = __ldg(l1 + j + 1);
                }
                const float top = __fmaf_rn(wa1, __fsub_rn(v01, v00), v00);
                const float bot = __fmaf_rn(wa1, __fsub_rn(v11, v10), v10);
                acc1 = __fadd_rn(acc1, __fmaf_rn(wz1, __fsub_rn(bot, top), top));
            }
            lk += PAR ? 2 * smaj : smaj;
            tk += PAR ? 2.0f : 1.0f;
        }
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            float a0, a1;
            unpack2(acc[r], a0, a1);
            fwd_sum[(64 * r + lane) * (ncol + 1) + threadIdx.y] = a0;
            fwd_sum[(64 * r + 32 + lane) * (ncol + 1) + threadIdx.y] = a1;
        }
        if (R & 1) fwd_sum[(32 * (R - 1) + lane) * (ncol + 1) + threadIdx.y] = acc1;
    }
    __syncthreads();
    double sq = 0.0;
    for (int i = threadIdx.y * 32 + lane; i < 32 * R * ncol; i += 32 * ncol) {
        const int cu = i % ncol, row = i / ncol, iv = iv0 + row, ju = iu0 + cu;
        if (iv >= d.nv || ju >= d.nu) continue;
        const float step = ray_z(load_col(col, (size_t)g * d.nu + ju), det_v(iv, d), d.cz).step;
        float* sum = fwd_sum + row * (ncol + 1) + cu;
        const float val = *sum * step;
        const size_t ray = ((size_t)g * d.nv + iv) * d.nu + ju;
        float res = val;
        if (MODE == FWD_LAMBDA) res = step * (lam[ray] * val);
        if (MODE == FWD_RESIDUAL) res = step * (lam[ray] * (meas[ray] - val));
        if (MODE == FWD_ICD) {
            sq += (double)lam[ray] * (double)val * (double)val;
            res = __fmul_rn(__fmul_rn(step, lam[ray]), val);
        }
        if (ROWS) *sum = res;
        else out[ray] = res;
    }
    if (ROWS) {
        __syncthreads();
        float* o = out + ((size_t)g * d.nu + iu) * sino_pitch(d.nv) + SINO_FRONT;
        for (int row = lane; iu < d.nu && row < 32 * R && iv0 + row < d.nv; row += 32)
            o[iv0 + row] = fwd_sum[row * (ncol + 1) + threadIdx.y];
    }
    if (MODE == FWD_ICD) {
        const double sum = block_sum_f64(sq);
        icd_alpha(sum, t, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y, S);
    }
}

// ------------------------------------------------------------------ adjoint (gather)

constexpr int ADJ_T = 4;           // a block's tile: ADJ_T x ADJ_T voxel lines in (x, y), one warp per ADJ_T
constexpr int ADJ_ENTRIES = 32;    // columns of a warp's list
// floats of one line in a block's tile: its 32 J voxels, and 8 that put the
// lines read together on different banks
__host__ __device__ constexpr int adj_line(int J) { return 32 * J + 8; }

// One detector column that crosses a warp's run of voxel lines; what the packed
// operations take is stored twice.
struct __align__(16) AdjEntry {
    float2 dfz, nrdfz;   // row spacing along z on this plane (voxels), and minus its reciprocal
    float2 c0, wa;       // cv + 1 - 1/dfz; weight of the line after the crossing
    float2 wb;           // 1 - wa: weight of the line before it
    const float* row0;   // the column's row 0, less FLOOR_MAGIC_BITS elements
};
// slot flags: two or three rows per footprint, no window outside the line's margins
constexpr int ADJ_TWO = 32, ADJ_THREE = 16;

__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ f32x2 vfma(f32x2 a, f32x2 b, f32x2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ f32x2 vadd(f32x2 a, f32x2 b) { return add2(a, b); }
__device__ __forceinline__ float vadd_rd(float a, float b) { return __fadd_rd(a, b); }
__device__ __forceinline__ f32x2 vadd_rd(f32x2 a, f32x2 b) { return add2_rd(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ f32x2 vsub(f32x2 a, f32x2 b) { return sub2(a, b); }
template <typename V> struct Lanes;
template <> struct Lanes<float> {
    static constexpr int N = 1;
    __device__ static __forceinline__ float all(float a) { return a; }
    __device__ static __forceinline__ float pack(const float* a) { return a[0]; }
    __device__ static __forceinline__ void unpack(float v, float* a) { a[0] = v; }
};
template <> struct Lanes<f32x2> {
    static constexpr int N = 2;
    __device__ static __forceinline__ f32x2 all(float a) { return pack2(a, a); }
    __device__ static __forceinline__ f32x2 pack(const float* a) { return pack2(a[0], a[1]); }
    __device__ static __forceinline__ void unpack(f32x2 v, float* a) { unpack2(v, a[0], a[1]); }
};

__device__ __forceinline__ float vbc(float2 a, float) { return a.x; }
__device__ __forceinline__ f32x2 vbc(float2 a, f32x2) { return pack2(a.x, a.y); }

// sum over the rows iv of one column of max(0, 1 - |f_z(iv) - z|) e'(iv) for
// the voxels V of a lane (one, or two packed).  f_z(iv) - z = (iv - cv) dfz +
// (cz - z), both bracketed terms exact, so only dfz carries a rounding.  The
// window starts at the first row with f_z > z - 1 and holds NR rows (NR = 0:
// `rows`, any number).  CLAMP: the window may lie outside the detector, and hold
// more rows than a footprint (2 / dfz, rounded up); otherwise all rows but its
// last lie inside the footprint.  A row outside it is dropped, so that a
// non-finite reading reaches the voxels of its own footprint only.  SQ: squared
// weights.
template <int NR, bool CLAMP, bool SQ, typename V>
__device__ __forceinline__ V row_sum(const AdjEntry& q, int rows, V zc, const ProjDims& d) {
    using L = Lanes<V>;
    float lo[L::N], w[L::N], ev[L::N];
    const V dfz = vbc(q.dfz, V());
    V t = vfma(zc, vbc(q.nrdfz, V()), vbc(q.c0, V()));
    if (CLAMP) {
        float tt[L::N];
        L::unpack(t, tt);
#pragma unroll
        for (int k = 0; k < L::N; ++k) tt[k] = fminf(fmaxf(tt[k], (float)-SINO_FRONT), (float)d.nv);
        t = L::pack(tt);
    }
    const V m = vadd_rd(t, L::all(FLOOR_MAGIC));
    const V iv = vsub(m, L::all(FLOOR_MAGIC));
    V df = vfma(vsub(iv, L::all(d.cv)), dfz, zc);
    L::unpack(m, lo);
    V s = L::all(0.0f);
    const int n = NR ? NR : rows;
#pragma unroll(NR ? NR : 1)
    for (int i = 0; i < n; ++i) {
        float dd[L::N];
        L::unpack(df, dd);
#pragma unroll
        for (int k = 0; k < L::N; ++k) {
            const int row = __float_as_int(lo[k]) + i;
            w[k] = __saturatef(__fsub_rn(1.0f, fabsf(dd[k])));
            if (SQ) w[k] = __fmul_rn(w[k], w[k]);
            if (NR) ev[k] = __ldg(q.row0 + row);
            else ev[k] = (unsigned)(row - FLOOR_MAGIC_BITS) < (unsigned)d.nv ? __ldg(q.row0 + row) : 0.0f;
            if (i == n - 1 || CLAMP) ev[k] = w[k] > 0.0f ? ev[k] : 0.0f;
        }
        s = vfma(L::pack(w), L::pack(ev), s);
        if (i + 1 < n) df = vadd(df, dfz);
    }
    return s;
}

// The gather's sums of J voxels per lane: J / 2 pairs, and one alone if J is odd.
template <int J>
struct AdjAcc {
    f32x2 p[J / 2 + 1];
    float o;
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < J / 2; ++j) p[j] = 0;
        o = 0.0f;
    }
    __device__ __forceinline__ void add(float2 w, const AdjAcc& s) {
#pragma unroll
        for (int j = 0; j < J / 2; ++j) p[j] = fma2(pack2(w.x, w.y), s.p[j], p[j]);
        if (J & 1) o = __fmaf_rn(w.x, s.o, o);
    }
    __device__ __forceinline__ void get(float* v) const {
#pragma unroll
        for (int j = 0; j < J / 2; ++j) unpack2(p[j], v[2 * j], v[2 * j + 1]);
        if (J & 1) v[J - 1] = o;
    }
    __device__ __forceinline__ void set(const float* v) {
#pragma unroll
        for (int j = 0; j < J / 2; ++j) p[j] = pack2(v[2 * j], v[2 * j + 1]);
        if (J & 1) o = v[J - 1];
    }
};

template <int NR, bool CLAMP, bool SQ, int J>
__device__ __forceinline__ void row_sums(const AdjEntry& q, int rows, const AdjAcc<J>& zc, const ProjDims& d,
                                         AdjAcc<J>& s) {
#pragma unroll
    for (int j = 0; j < J / 2; ++j) s.p[j] = row_sum<NR, CLAMP, SQ, f32x2>(q, rows, zc.p[j], d);
    if (J & 1) s.o = row_sum<NR, CLAMP, SQ, float>(q, rows, zc.o, d);
}

// Adds to the ADJ_T voxel lines a_lo, a_lo + STR, ... of plane kpl (x for
// x-major rays, else y) the terms of every ray whose major axis is XMAJ.  STR = 2
// takes the voxels of one parity (the ICD agent's groups: also along z, which zc
// carries), of whose lines a column touches one; SQ takes squared weights (the
// diagonal of A^T Lambda A, with e = step^2 Lambda).
//
// A column's ray plane crosses the voxel plane at f_a between the lines a0 and
// a0 + 1, to which it adds (1 - w_a) s and w_a s with the same sums s over its
// rows.  The lanes first build a list: `slots` columns of 32 / slots views at a
// time (adj_slots: about as many as a run has), those that the projection of the
// run's ends brackets (with a margin far above that projection's rounding) and
// whose f_a, formed with the forward's own operations (bit for bit), touches the
// run.  The warp then walks the list, its lanes taking voxels along z.  The order
// of a voxel's terms (groups of views, columns in each) does not depend on J.
// Part `part` of `parts` takes every parts-th group of views.
template <bool XMAJ, int J, int STR, bool SQ>
__device__ __forceinline__ void gather_run(const float4* __restrict__ col, const float2* __restrict__ trig,
                                           const int* __restrict__ vflag, const float* __restrict__ e, int t, int kpl,
                                           int a_lo, int z_lo, const AdjAcc<J>& zc, const ProjDims& d, int slots, int part,
                                           int parts, AdjEntry* __restrict__ list, int* __restrict__ slot,
                                           AdjAcc<J>* acc) {
    const int lane = threadIdx.x;
    const int na = XMAJ ? d.ny : d.nx, nvp = sino_pitch(d.nv);
    const int a_hi = min(a_lo + STR * (ADJ_T - 1) + 1, na);
    const float tk = __fsub_rn((float)kpl, XMAJ ? d.cx : d.cy);
    const float maj = tk * d.vox, lo = (a_lo - 1 - (XMAJ ? d.cy : d.cx)) * d.vox, hi = (a_hi - (XMAJ ? d.cy : d.cx)) * d.vox;
    const float margin = 0.01f + 4e-6f * d.nu;
    // views of a group: as many as the lanes take, but no fewer groups than parts
    const int vstep = min(32 / slots, (d.views + parts - 1) / parts), vi = lane / slots, ci = lane - vi * slots;
    for (int v0 = part * vstep; v0 < d.views; v0 += parts * vstep) {
        const int v = v0 + vi, g = t * d.views + v;
        int iu = d.nu, iu_hi = -1, flags = 0;
        float2 cs = make_float2(0.0f, 0.0f);
        if (vi < vstep && v < d.views) {
            flags = __ldg(vflag + g);
            cs = __ldg(trig + g);
        }
        if (flags & (XMAJ ? 1 : 2)) {
            const float x1 = XMAJ ? maj : lo, y1 = XMAJ ? lo : maj, x2 = XMAJ ? maj : hi, y2 = XMAJ ? hi : maj;
            // an end beside the source projects anywhere: try every column
            const bool near = fminf(d.dso - x1 * cs.x - y1 * cs.y, d.dso - x2 * cs.x - y2 * cs.y) < 0.05f * d.dso;
            const float u1 = u_pixel(x1, y1, cs.x, cs.y, d), u2 = u_pixel(x2, y2, cs.x, cs.y, d);
            iu = (near ? 0 : max(0, (int)ceilf(fminf(u1, u2) - margin))) + ci;
            iu_hi = near ? d.nu - 1 : min(d.nu - 1, (int)floorf(fmaxf(u1, u2) + margin));
        }
        while (__any_sync(0xffffffffu, iu <= iu_hi)) {
            bool ok = iu <= iu_hi;
            AdjEntry q;
            int al = 0, fast = 0;
            if (ok) {
                const size_t gcol = (size_t)g * d.nu + iu;
                const float4 c = __ldg(col + 2 * gcol);   // fa_mid, ba, c1, inv_dmaj
                if (flags == 3) ok = (__ldg(col + 2 * gcol + 1).z != 0.0f) == XMAJ;
                const float fa = __fmaf_rn(tk, c.y, c.x);
                const float a0f = floorf(fa);
                float wa = __fsub_rn(fa, a0f), wb = __fsub_rn(1.0f, wa);
                al = (int)a0f - a_lo;
                ok = ok && al >= -1;
                if (STR == 2) {   // the line of the group beside the crossing
                    if (!(al & 1)) wa = wb;
                    al = (al + 1) >> 1;
                }
                ok = ok && al < ADJ_T;
                if (SQ) wa = __fmul_rn(wa, wa), wb = __fmul_rn(wb, wb);
                const float dfz = d.dv * __fmaf_rn(tk, c.w, c.z), rdfz = __fdividef(1.0f, dfz);
                const float c0 = d.cv + 1.0f - rdfz;
                q.dfz = make_float2(dfz, dfz);
                q.nrdfz = make_float2(-rdfz, -rdfz);
                q.c0 = make_float2(c0, c0);
                q.wa = make_float2(wa, wa);
                q.wb = make_float2(wb, wb);
                q.row0 = e + gcol * nvp + SINO_FRONT - FLOOR_MAGIC_BITS;
                // every window of the run's voxels inside the line's margins
                const float t_lo = __fmaf_rn(d.cz - (float)z_lo, -rdfz, c0);
                const float t_hi = __fmaf_rn(d.cz - (float)min(z_lo + STR * (32 * J - 1), d.nz - 1), -rdfz, c0);
                if (t_lo > 1.0f - SINO_FRONT && t_hi < (float)d.nv)
                    fast = rdfz > 0.5f && rdfz <= 1.0f ? ADJ_TWO : rdfz > 1.0f && rdfz <= 1.5f ? ADJ_THREE : 0;
            }
            const unsigned mask = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const int at = __popc(mask & ((1u << lane) - 1));
                list[at] = q;
                slot[at] = (al & 7) | fast;
            }
            __syncwarp();
            const int n = __popc(mask);
            for (int i = 0; i < n; ++i) {
                const AdjEntry q = list[i];
                const int sl = slot[i];
                AdjAcc<J> s;
                if (sl >= ADJ_TWO) {
                    row_sums<2, false, SQ, J>(q, 0, zc, d, s);
                } else if (sl >= ADJ_THREE) {
                    row_sums<3, false, SQ, J>(q, 0, zc, d, s);
                } else {
                    const float span = -2.0f * q.nrdfz.x;   // rows per footprint: ceil(2 / dfz)
                    if (span <= 3.0f) row_sums<3, true, SQ, J>(q, 0, zc, d, s);
                    else row_sums<0, true, SQ, J>(q, (int)fminf(ceilf(span), (float)(d.nv + 8)), zc, d, s);
                }
                if (STR == 2) {
                    switch (sl & 7) {
                        case 0: acc[0].add(q.wa, s); break;
                        case 1: acc[1].add(q.wa, s); break;
                        case 2: acc[2].add(q.wa, s); break;
                        default: acc[3].add(q.wa, s); break;
                    }
                } else switch (sl & 7) {
                    case 7: acc[0].add(q.wa, s); break;   // -1: the line before the run
                    case 0: acc[0].add(q.wb, s); acc[1].add(q.wa, s); break;
                    case 1: acc[1].add(q.wb, s); acc[2].add(q.wa, s); break;
                    case 2: acc[2].add(q.wb, s); acc[3].add(q.wa, s); break;
                    default: acc[3].add(q.wb, s); break;
                }
            }
            __syncwarp();
            iu += slots;
        }
    }
}

// Blocks per SM that the register limit asks for, by A^T's time with 1 (no limit) / 4 / 5 / 6 / 8 of
// them (us, 24 views): J = 1 (256^2 x 32 x 8) 1089-1094 with any; J = 2 (128^2 x 64 x 8) 327 / 327 / 328 /
// 295 / 279; J = 3 (128^2 x 96 x 8) 401 / 401 / 368 / 348 / 348; J = 4 (128^3 x 8) 449 / 449 / 452 / 420 /
// 416; J = 5 (160^3 x 4) 426 / 424 / 385 / 377 / 392; J = 6 (192^3 x 4) 649 / 640 / 582 / 605 / 614; J = 8
// (256^3 x 2) 773 / 665 / 663 / 697 / 806; J = 10 (320^3) 699 / 636 / 692 / 731 / 964; J = 12 (384^3 x 2) 2768 /
// 2076 / 2185 / 2519 / 3424 (with 3: 2164).
__host__ __device__ constexpr int adj_min_blocks(int J) { return J >= 8 ? 4 : J >= 5 ? 5 : J >= 3 ? 6 : 8; }

// Both phases of a block on the lines x0 + STR i, y0 + STR w, voxels z_lo + STR (lane
// + 32 j): leaves in acc[i] the sums of the lines of y = y0 + STR w (none if that
// lies outside the volume).  VS sets of ADJ_T warps share the views (a small
// volume has too few tiles to fill the GPU, and a warp's walk over the views sets
// its time); the first set holds the result.
template <int J, int VS>
struct AdjShared {
    AdjEntry list[ADJ_T * VS][ADJ_ENTRIES];
    int slot[ADJ_T * VS][ADJ_ENTRIES];
};

template <int J, int VS, int STR, bool SQ>
__device__ __forceinline__ void gather_tile(const float4* __restrict__ col, const float2* __restrict__ trig,
                                            const int* __restrict__ vflag, const float* __restrict__ e, int t, int x0,
                                            int y0, int z_lo, const ProjDims& d, int slots, float* adj_tile,
                                            AdjShared<J, VS>& sh, AdjAcc<J>* acc) {
    const int lane = threadIdx.x, wv = threadIdx.y, w = VS == 1 ? wv : wv % ADJ_T, part = VS == 1 ? 0 : wv / ADJ_T;
    AdjAcc<J> zc;
    {
        float a[J];   // voxels past the volume repeat its last one
#pragma unroll
        for (int j = 0; j < J; ++j) a[j] = d.cz - (float)min(z_lo + STR * (lane + 32 * j), d.nz - 1);
        zc.set(a);
    }
    float* all = adj_tile + part * ADJ_T * ADJ_T * adj_line(J);
    float* tile = all + w * ADJ_T * adj_line(J);   // the lines of y = y0 + STR w
    auto put = [&](float* line, int stride) {
#pragma unroll
        for (int i = 0; i < ADJ_T; ++i) {
            float v[J];
            acc[i].get(v);
#pragma unroll
            for (int j = 0; j < J; ++j) line[i * stride + 32 * j + lane] = v[j];
        }
    };
#pragma unroll
    for (int i = 0; i < ADJ_T; ++i) acc[i].zero();
    if (x0 + STR * w < d.nx)
        gather_run<true, J, STR, SQ>(col, trig, vflag, e, t, x0 + STR * w, y0, z_lo, zc, d, slots, part, VS, sh.list[wv],
                                     sh.slot[wv], acc);
    put(all + w * adj_line(J), ADJ_T * adj_line(J));
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ADJ_T; ++i) {
        float v[J];
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] = tile[i * adj_line(J) + 32 * j + lane];
        acc[i].set(v);
    }
    if (y0 + STR * w < d.ny)
        gather_run<false, J, STR, SQ>(col, trig, vflag, e, t, y0 + STR * w, x0, z_lo, zc, d, slots, part, VS, sh.list[wv],
                                      sh.slot[wv], acc);
    if (VS > 1) {   // the parts' sums in order
        if (part > 0) put(tile, adj_line(J));
        __syncthreads();
        if (part > 0) return;
#pragma unroll
        for (int i = 0; i < ADJ_T; ++i) {
            float v[J];
            acc[i].get(v);
            for (int k = 1; k < VS; ++k)
#pragma unroll
                for (int j = 0; j < J; ++j)
                    v[j] = __fadd_rn(v[j], tile[(k * ADJ_T * ADJ_T + i) * adj_line(J) + 32 * j + lane]);
            acc[i].set(v);
        }
    }
}

// A block takes ADJ_T x ADJ_T voxel lines and 32 J voxels of each; lane = z, so
// that a warp's loads run along the detector rows.  First warp w takes the lines
// of x = x0 + w for the x-major rays, then, the sums handed over through shared
// memory, those of y = y0 + w for the y-major rays: either way a column's sums
// over its rows, most of the work, serve both lines beside its crossing, and no
// sum is read back per ray.  Bound by instruction issue: about 14 instructions
// per (column, voxel along z), and some 40 per column that J voxels per lane
// share (packed pairs, the list, the choice of the two lines).  A thread per run
// of voxels that added each row's two terms into shared memory visited every
// crossing twice: A^T at 384^3 x 16, 512 x 384, 24 views 41.6 -> 14.3 ms (J = 12;
// J = 4: 18.5), 128^3 x 8, 192 x 160, 32 views in a 90 degree wedge 1.59 -> 0.63
// ms, 24^3 x 4, 32 x 32, 12 views 85 -> 30 us.  Tiles of 8 x 8 lines with J = 4
// need fewer columns per line (0.79 against 0.88) but took 20 ms.
// e is the step-weighted sinogram e' = step * e in lines of rows.
//   ADJ_PLAIN:   out = A^T e
//   ADJ_CG_INIT: r = A^T e + (v - z)/sigma^2, p = r, rr = r.r (a1 = v - z)
//   ADJ_CG_Q:    q = A^T e + p/sigma^2, alpha = rr / p.q      (a1 = p)
//   ADJ_THETA2:  (A.^2)^T e + 1/sigma^2 (the ICD agent's curvature)
// (the CG's vectors as lines, the volume of ADJ_PLAIN as [nt][nz][ny][nx])
template <int MODE, int J, int VS>
__global__ void __launch_bounds__(32 * ADJ_T * VS, adj_min_blocks(J) >= VS ? adj_min_blocks(J) / VS : 1) joseph_adj_kernel(
    const float4* __restrict__ col, const float2* __restrict__ trig, const int* __restrict__ vflag,
    const float* __restrict__ e, float* __restrict__ out, const float* __restrict__ a1, float* __restrict__ out2,
    CgScalars cg, float inv_s2, ProjDims d, int slots) {
    extern __shared__ float adj_tile[];   // [y][x][adj_line(J)]
    __shared__ AdjShared<J, VS> sh;
    const int lane = threadIdx.x, w = threadIdx.y;
    const int nzb = (d.nz + 32 * J - 1) / (32 * J);
    const int zb = blockIdx.z % nzb, t = blockIdx.z / nzb;
    const int x0 = blockIdx.x * ADJ_T, y0 = blockIdx.y * ADJ_T, z0 = zb * 32 * J + lane;
    if (MODE == ADJ_CG_INIT || MODE == ADJ_CG_Q) {
        // the vector that the epilogue reads, into L2: with 16 warps on an SM
        // nothing else would hide its way from memory (19.5 -> 18.1 ms, A^T in the CG
        // at 384^3 x 16)
        const size_t first = (((size_t)t * d.ny + y0 + w) * d.nx + x0) * vz_pitch(d.nz) + VZ_FRONT + zb * 32 * J;
        for (int k = lane; k < ADJ_T * J && w < ADJ_T && y0 + w < d.ny; k += 32)
            if (x0 + k / J < d.nx && zb * 32 * J + k % J * 32 < d.nz)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a1 + first + (size_t)(k / J) * vz_pitch(d.nz) + k % J * 32));
    }
    AdjAcc<J> acc[ADJ_T];
    gather_tile<J, VS, 1, MODE == ADJ_THETA2>(col, trig, vflag, e, t, x0, y0, zb * 32 * J, d, slots, adj_tile, sh, acc);
    float* tile = adj_tile + w * ADJ_T * adj_line(J);
    const int iy = y0 + w;
    double dot = 0.0;
    if (w < ADJ_T && iy < d.ny) {
        if (MODE == ADJ_PLAIN) {
            // the volume is contiguous along x: ADJ_T lanes write the x of one z
#pragma unroll
            for (int i = 0; i < ADJ_T; ++i) {
                float v[J];
                acc[i].get(v);
#pragma unroll
                for (int j = 0; j < J; ++j) tile[i * adj_line(J) + 32 * j + lane] = v[j];
            }
            __syncwarp();
            const int ix = x0 + lane % ADJ_T;
#pragma unroll 4
            for (int k = lane / ADJ_T; k < 32 * J; k += 32 / ADJ_T) {
                const int iz = zb * 32 * J + k;
                if (ix >= d.nx || iz >= d.nz) break;
                out[(((size_t)t * d.nz + iz) * d.ny + iy) * d.nx + ix] = tile[(lane % ADJ_T) * adj_line(J) + k];
            }
        } else {
            const int nzp = vz_pitch(d.nz);
            const size_t first = (((size_t)t * d.ny + iy) * d.nx + x0) * nzp + VZ_FRONT + z0;
#pragma unroll
            for (int i = 0; i < ADJ_T; ++i) {
                if (x0 + i >= d.nx) break;
                float v[J];
                acc[i].get(v);
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    if (z0 + 32 * j >= d.nz) break;
                    const size_t k = first + i * nzp + 32 * j;
                    if (MODE == ADJ_THETA2) {
                        out[k] = v[j] + inv_s2;
                        continue;
                    }
                    const float a = a1[k], r = __fmaf_rn(a, inv_s2, v[j]);
                    out[k] = r;
                    if (MODE == ADJ_CG_INIT) out2[k] = r;
                    dot += (double)(MODE == ADJ_CG_INIT ? r : a) * (double)r;
                }
            }
        }
    }
    if (MODE == ADJ_CG_INIT || MODE == ADJ_CG_Q) {
        const double sum = block_sum_f64(dot);
        const int bpf = gridDim.x * gridDim.y * nzb;   // blocks per frame
        const int b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * zb);
        frame_finalize<MODE == ADJ_CG_INIT ? FIN_RR0 : FIN_ALPHA>(sum, t, b, bpf, cg);
    }
}

// e' = step * e for every ray, into lines of rows (the gather's input), through
// 32 x 32 tiles of one view.
__global__ void step_weight_kernel(const float4* __restrict__ col, const float* __restrict__ e,
                                   float* __restrict__ out, ProjDims d) {
    __shared__ float tile[32][33];
    const int g = blockIdx.x, u0 = blockIdx.y * 32, v0 = blockIdx.z * 32;
    const int iu = u0 + threadIdx.x;
    if (iu < d.nu) {
        const ColParams c = load_col(col, (size_t)g * d.nu + iu);
        for (int k = threadIdx.y; k < 32 && v0 + k < d.nv; k += blockDim.y)
            tile[k][threadIdx.x] = ray_z(c, det_v(v0 + k, d), d.cz).step * e[((size_t)g * d.nv + v0 + k) * d.nu + iu];
    }
    __syncthreads();
    const int iv = v0 + threadIdx.x;
    if (iv >= d.nv) return;
    for (int k = threadIdx.y; k < 32 && u0 + k < d.nu; k += blockDim.y)
        out[((size_t)g * d.nu + u0 + k) * sino_pitch(d.nv) + SINO_FRONT + iv] = tile[threadIdx.x][k];
}

// ------------------------------------------------------------------ CG vectors

// Walks lines of n values (pitch apart, a margin of VZ_FRONT = SINO_FRONT before
// them): a warp of the `blocks` blocks takes one line (several short ones), its
// lanes units of four values.  The margins of the lines stay untouched.
static_assert(VZ_FRONT == 4 && SINO_FRONT == 4, "for_units: units of four values start on 16 bytes");
template <typename L, typename F>
__device__ __forceinline__ void for_units(size_t lines, int n, int pitch, int block, int blocks, L&& line, F&& f) {
    const int n4 = (n + 3) / 4;
    int gw = 32;   // lanes per line
    while (gw > 1 && gw / 2 >= n4) gw /= 2;
    const int lane = threadIdx.x & 31, per = 32 / gw, warps = blockDim.x >> 5;
    const size_t first = ((size_t)block * warps + (threadIdx.x >> 5)) * per + lane / gw;
    for (size_t l = first; l < lines; l += (size_t)blocks * warps * per) {
        const size_t at = (size_t)line(l) * pitch + VZ_FRONT;
        for (int u = lane % gw; u < n4; u += gw) f(at + 4 * u, min(4, n - 4 * u));
    }
}
template <typename F>
__device__ __forceinline__ void for_voxels(size_t lines, int nz, F&& f) {
    for_units(lines, nz, vz_pitch(nz), blockIdx.x, gridDim.x, [](size_t l) { return l; }, f);
}

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
// the first n of four values
__device__ __forceinline__ void store4(float* p, float4 v, int n) {
    if (n == 4) {
        *reinterpret_cast<float4*>(p) = v;
    } else {
        p[0] = v.x;
        if (n > 1) p[1] = v.y;
        if (n > 2) p[2] = v.z;
    }
}
__device__ __forceinline__ float4 fma4(float a, float4 x, float4 y) {
    return make_float4(__fmaf_rn(a, x.x, y.x), __fmaf_rn(a, x.y, y.y), __fmaf_rn(a, x.z, y.z), __fmaf_rn(a, x.w, y.w));
}

// r -= alpha q; beta = r.r / rr  (grid: blocks of a frame x nt).  Each thread
// adds the squares of runs of 8 of its elements in FP32 before its FP64 sum
// (FP64 arithmetic is a small fraction of the FP32 rate on this GPU); the order
// of every addition is fixed.  Bound by HBM (12 bytes per voxel).
__global__ void __launch_bounds__(256) cg_residual_kernel(float* __restrict__ r, const float* __restrict__ q,
                                                          const double* __restrict__ alpha, CgScalars cg, size_t lines,
                                                          int nz) {
    const int t = blockIdx.y;
    const float a = -(float)alpha[t];
    const size_t off = (size_t)t * lines * vz_pitch(nz);
    double dot = 0.0;
    float run = 0.0f;
    int k = 0;
    for_voxels(lines, nz, [&](size_t i, int n) {
        const float4 v = fma4(a, load4(q + off + i), load4(r + off + i));
        store4(r + off + i, v, n);
        run = __fmaf_rn(v.x, v.x, run);
        if (n > 1) run = __fmaf_rn(v.y, v.y, run);
        if (n > 2) run = __fmaf_rn(v.z, v.z, run);
        if (n > 3) run = __fmaf_rn(v.w, v.w, run);
        if (++k & 1) return;
        dot += (double)run;
        run = 0.0f;
    });
    const double s = block_sum_f64(dot + (double)run);
    frame_finalize<FIN_BETA>(s, t, blockIdx.x, gridDim.x, cg);
}

// z += alpha p; p = r + beta p.  Bound by HBM (20 bytes per voxel).
__global__ void __launch_bounds__(256) cg_direction_kernel(float* __restrict__ z, float* __restrict__ p,
                                                           const float* __restrict__ r,
                                                           const double* __restrict__ alpha,
                                                           const double* __restrict__ beta, size_t lines, int nz) {
    const int t = blockIdx.y;
    const float a = (float)alpha[t], b = (float)beta[t];
    const size_t off = (size_t)t * lines * vz_pitch(nz);
    for_voxels(lines, nz, [&](size_t i, int n) {
        const float4 pv = load4(p + off + i);
        store4(z + off + i, fma4(a, pv, load4(z + off + i)), n);
        store4(p + off + i, fma4(b, pv, load4(r + off + i)), n);
    });
}

// ------------------------------------------------------------------ grouped ICD data agent
//
// The partial update L~ of Sec. III as coordinate descent on the cost of
// Eq. (4).  A sweep visits the eight parity groups (pz*2 + py)*2 + px of the
// voxels in increasing order; inside a group every voxel takes its own Newton
// step against the same step-weighted residual sinogram e' = step*Lambda*(y - Az),
//     delta_s = -theta1_s / theta2_s,
//     theta1_s = -(A^T Lambda e)_s + (z_s - v_s)/sigma^2,
//     theta2_s = sum_r Lambda_r a_rs^2 + 1/sigma^2,
// and the group moves by alpha_t delta (per frame t), alpha_t the exact
// minimiser of the quadratic cost along delta.  A parity group holds at most
// one of the four bilinear taps of any ray-plane crossing.

// The group step's gather: for every voxel s of the group, delta_s =
// -theta1_s/theta2_s, and per-block partial sums of theta1.delta and delta.delta.
// All volumes as lines; delta is written for both z parities (zero for the other),
// so that the lines of the group hold this step's delta alone.  Tiles as in
// joseph_adj_kernel, in voxels of the group: 314 -> 89 us at 96^3 x 6, 160 x 128, 24
// views; with delta projected straight from its lines, the line search's sum in
// that projection and both updates in one launch, three sweeps 14.7 -> 5.8 ms.
template <int J, int VS>
__global__ void __launch_bounds__(32 * ADJ_T * VS, adj_min_blocks(J) >= VS ? adj_min_blocks(J) / VS : 1) icd_group_kernel(
    const float4* __restrict__ col, const float2* __restrict__ trig, const int* __restrict__ vflag,
    const float* __restrict__ e, const float* __restrict__ z, const float* __restrict__ v,
    const float* __restrict__ theta2, float* __restrict__ dlt, IcdSums S, float inv_s2, IcdGroup G, ProjDims d,
    int slots) {
    extern __shared__ float adj_tile[];
    __shared__ AdjShared<J, VS> sh;
    const int lane = threadIdx.x, w = threadIdx.y;
    const int pairs = (d.nz + 1) / 2, nzb = (pairs + 32 * J - 1) / (32 * J);
    const int zb = blockIdx.z % nzb, t = blockIdx.z / nzb;
    const int x0 = G.px + 2 * ADJ_T * blockIdx.x, y0 = G.py + 2 * ADJ_T * blockIdx.y, m0 = zb * 32 * J;
    AdjAcc<J> acc[ADJ_T];
    gather_tile<J, VS, 2, false>(col, trig, vflag, e, t, x0, y0, G.pz + 2 * m0, d, slots, adj_tile, sh, acc);
    const int iy = y0 + 2 * w, nzp = vz_pitch(d.nz);
    double gd = 0.0, dd = 0.0;
    if (w < ADJ_T && iy < d.ny) {
        const size_t first = (((size_t)t * d.ny + iy) * d.nx + x0) * nzp + VZ_FRONT;
#pragma unroll
        for (int i = 0; i < ADJ_T; ++i) {
            if (x0 + 2 * i >= d.nx) break;
            float a[J];
            acc[i].get(a);
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = m0 + lane + 32 * j;
                if (m >= pairs) break;
                const size_t k = first + 2 * i * nzp + 2 * m;
                float del = 0.0f;
                if (2 * m + G.pz < d.nz) {
                    const float th1 = __fmaf_rn(__fsub_rn(z[k + G.pz], v[k + G.pz]), inv_s2, -a[j]);
                    del = -__fdiv_rn(th1, theta2[k + G.pz]);
                    gd += (double)th1 * (double)del;
                    dd += (double)del * (double)del;
                }
                *reinterpret_cast<float2*>(dlt + k) = G.pz ? make_float2(0.0f, del) : make_float2(del, 0.0f);
            }
        }
    }
    gd = block_sum_f64(gd);
    dd = block_sum_f64(dd);
    if (lane == 0 && w == 0) {
        double* out = S.gpart + 2 * ((size_t)t * S.gblocks + blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * zb));
        out[0] = gd;
        out[1] = dd;
    }
}

// After a group step: e' -= alpha_t ad, ad = step Lambda (A delta), over the sinogram's
// lines of rows (the first half of a frame's blocks), z += alpha_t delta over the
// group's lines (the second half).
__global__ void __launch_bounds__(256) icd_update_kernel(float* __restrict__ e, const float* __restrict__ ad,
                                                         float* __restrict__ z,
                                                         const float* __restrict__ dlt,
                                                         const double* __restrict__ alpha, IcdGroup G, ProjDims d) {
    const int t = blockIdx.y, half = gridDim.x / 2;
    const float a = (float)alpha[t];
    if (blockIdx.x < half) {
        const size_t lines = (size_t)d.views * d.nu, off = (size_t)t * lines * sino_pitch(d.nv);
        for_units(lines, d.nv, sino_pitch(d.nv), blockIdx.x, half, [&](size_t l) { return l; }, [&](size_t i, int n) {
            store4(e + off + i, fma4(-a, load4(ad + off + i), load4(e + off + i)), n);
        });
    } else {
        const size_t off = (size_t)t * d.ny * d.nx * vz_pitch(d.nz);
        for_units((size_t)G.gx * G.gy, d.nz, vz_pitch(d.nz), blockIdx.x - half, half,
                  [&](size_t l) { return (2 * (l / G.gx) + G.py) * d.nx + 2 * (l % G.gx) + G.px; },
                  [&](size_t i, int n) { store4(z + off + i, fma4(a, load4(dlt + off + i), load4(z + off + i)), n); });
    }
}

// e2 = step^2 Lambda (the theta2 gather's input) as lines of rows, through 32 x 32
// tiles of one view.
__global__ void icd_weights_kernel(const float4* __restrict__ col, const float* __restrict__ lam,
                                   float* __restrict__ e2, ProjDims d) {
    __shared__ float tile[32][33];
    const int g = blockIdx.x, u0 = blockIdx.y * 32, v0 = blockIdx.z * 32;
    const int iu = u0 + threadIdx.x;
    if (iu < d.nu) {
        const ColParams c = load_col(col, (size_t)g * d.nu + iu);
        for (int k = threadIdx.y; k < 32 && v0 + k < d.nv; k += blockDim.y) {
            const float step = ray_z(c, det_v(v0 + k, d), d.cz).step;
            tile[k][threadIdx.x] = __fmul_rn(__fmul_rn(step, step), lam[((size_t)g * d.nv + v0 + k) * d.nu + iu]);
        }
    }
    __syncthreads();
    const int iv = v0 + threadIdx.x;
    if (iv >= d.nv) return;
    for (int k = threadIdx.y; k < 32 && u0 + k < d.nu; k += blockDim.y)
        e2[((size_t)g * d.nu + u0 + k) * sino_pitch(d.nv) + SINO_FRONT + iv] = tile[threadIdx.x][k];
}

// ------------------------------------------------------------------ phantom (test data)

#define MSF_MAX_ELL_RECORDS 256
__constant__ double c_ell[MSF_MAX_ELL_RECORDS * 16];

__device__ __forceinline__ void ell_local(const double* e, double px, double py, double pz,
                                          double* q) {
    const double tx = px - e[0], ty = py - e[1], tz = pz - e[2];
    for (int k = 0; k < 3; ++k)
        q[k] = (e[6 + 3 * k] * tx + e[7 + 3 * k] * ty + e[8 + 3 * k] * tz) / e[3 + k];
}

__global__ void phantom_voxelize_kernel(float* __restrict__ x, int nx, int ny, int nz, int nt,
                                        double vox, int n_ell, int ss) {
    const size_t fs = (size_t)nx * ny * nz;
    const size_t total = fs * nt;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(i / fs);
        size_t r = i % fs;
        const int iz = (int)(r / ((size_t)nx * ny));
        r %= (size_t)nx * ny;
        const int iy = (int)(r / nx), ix = (int)(r % nx);
        double acc = 0.0;
        for (int e = 0; e < n_ell; ++e) {
            const double* E = c_ell + 16 * ((size_t)t * n_ell + e);
            int inside = 0;
            for (int a = 0; a < ss; ++a)
                for (int b = 0; b < ss; ++b)
                    for (int cc = 0; cc < ss; ++cc) {
                        double q[3];
                        ell_local(E, (ix - 0.5 * (nx - 1) + (cc + 0.5) / ss - 0.5) * vox,
                                  (iy - 0.5 * (ny - 1) + (b + 0.5) / ss - 0.5) * vox,
                                  (iz - 0.5 * (nz - 1) + (a + 0.5) / ss - 0.5) * vox, q);
                        inside += (q[0] * q[0] + q[1] * q[1] + q[2] * q[2] <= 1.0);
                    }
            acc += E[15] * (double)inside / (double)(ss * ss * ss);
        }
        x[i] = (float)acc;
    }
}

__global__ void phantom_project_kernel(const double* __restrict__ angles, float* __restrict__ y,
                                       ProjDims d, double du, double dv, double dso, double dsd,
                                       int n_ell) {
    const size_t per_view = (size_t)d.nu * d.nv;
    const size_t total = per_view * d.views * d.nt;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int g = (int)(i / per_view);
        const int t = g / d.views;
        const int iv = (int)((i % per_view) / d.nu), iu = (int)(i % d.nu);
        const double th = angles[g], c = cos(th), s = sin(th);
        const double u = (iu - 0.5 * (d.nu - 1)) * du, v = (iv - 0.5 * (d.nv - 1)) * dv;
        const double sx = dso * c, sy = dso * s;
        const double dx = -(dsd - dso) * c - u * s - sx, dy = -(dsd - dso) * s + u * c - sy,
                     dz = v;
        const double len = sqrt(dx * dx + dy * dy + dz * dz);
        double acc = 0.0;
        for (int e = 0; e < n_ell; ++e) {
            const double* E = c_ell + 16 * ((size_t)t * n_ell + e);
            double q0[3], q1[3];
            ell_local(E, sx, sy, 0.0, q0);
            for (int k = 0; k < 3; ++k)
                q1[k] = (E[6 + 3 * k] * dx + E[7 + 3 * k] * dy + E[8 + 3 * k] * dz) / E[3 + k];
            const double A = q1[0] * q1[0] + q1[1] * q1[1] + q1[2] * q1[2];
            const double B = 2.0 * (q0[0] * q1[0] + q0[1] * q1[1] + q0[2] * q1[2]);
            const double C = q0[0] * q0[0] + q0[1] * q0[1] + q0[2] * q0[2] - 1.0;
            const double disc = B * B - 4.0 * A * C;
            if (disc > 0.0) acc += E[15] * len * sqrt(disc) / A;
        }
        y[i] = (float)acc;
    }
}

}  // namespace msf

// ====================================================================== handles

namespace msf {

static size_t vz_size(const msf_vol& v) {   // a volume as lines
    return VZ_FRONT + (size_t)v.nt * v.ny * v.nx * vz_pitch(v.nz);
}
static size_t rows_size(const msf_projector* p) {   // a sinogram in lines of rows
    return SINO_FRONT + (size_t)p->vol.nt * p->geom.views * p->geom.nu * sino_pitch(p->geom.nv);
}
// Whether the plan keeps lines and pairs in one place (some calls take either).
static bool shared_input(const msf_projector* p) { return p->d_vz && p->d_px; }

static dim3 lines_grid(const msf_vol& v) { return dim3((v.nx + LT - 1) / LT * v.ny * v.nt, (v.nz + LT - 1) / LT); }

static msf_status launch_lines(msf_projector* p, const float* in, cudaStream_t st) {
    const msf_vol& v = p->vol;
    MSF_PROF("transpose", st);
    lines_kernel<LINES_COPY><<<lines_grid(v), 256, 0, st>>>(in, p->d_vz, nullptr, nullptr, v.nx, v.ny, v.nz, shared_input(p));
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

// Detector columns (warps) per block of the forward; its row sets of 32 rows are
// split evenly over as few chunks as FWD_MAX_R allows.
static int fwd_cols(const msf_projector* p) { return p->fwd_bx / 8; }
static int fwd_chunks(const ProjDims& d) { return ((d.nv + 31) / 32 + FWD_MAX_R - 1) / FWD_MAX_R; }

template <int MODE, bool PAR, bool ROWS>
static void launch_fwd_kernel(msf_projector* p, const float* vz, float* out, const float* lam, const float* meas,
                              int kpx, int kpy, const IcdSums& S, cudaStream_t st) {
    const ProjDims& d = p->dims;
    const int ncol = fwd_cols(p);
    const int sets = (d.nv + 31) / 32, chunks = fwd_chunks(d), R = (sets + chunks - 1) / chunks;
    const dim3 block(32, ncol), grid((d.nu + ncol - 1) / ncol * d.views, chunks, d.nt);
    const size_t smem = (size_t)32 * R * (ncol + 1) * sizeof(float);
#define MSF_FWD_CASE(N)                                                                                            \
    case N:                                                                                                        \
        joseph_fwd_kernel<MODE, N, PAR, ROWS><<<grid, block, smem, st>>>(vz, p->d_zero, p->d_col, out, lam, meas, d,     \
                                                                    kpx, kpy, S);                                  \
        break;
    switch (R) {
        MSF_FWD_CASE(1)
        MSF_FWD_CASE(2)
        MSF_FWD_CASE(3)
        MSF_FWD_CASE(4)
        MSF_FWD_CASE(5)
    }
#undef MSF_FWD_CASE
}

// A of the volume whose lines are vz (MODE), written as a sinogram or, ROWS, as
// lines of rows.
template <int MODE, bool ROWS>
static msf_status launch_fwd_lines(msf_projector* p, const float* vz, float* out, const float* lam, const float* meas,
                                   cudaStream_t st) {
    MSF_PROF("joseph_fwd", st);
    launch_fwd_kernel<MODE, false, ROWS>(p, vz, out, lam, meas, 0, 0, IcdSums{}, st);
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

template <int MODE, bool ROWS>
static msf_status launch_fwd(msf_projector* p, const float* x, float* out, const float* lam, const float* meas,
                             cudaStream_t st) {
    MSF_TRY(launch_lines(p, x, st));
    return launch_fwd_lines<MODE, ROWS>(p, p->d_vz, out, lam, meas, st);
}

// Voxels per lane (J) of an adjoint launch: the plan's z-run allows at most 2 (8),
// 4 (16), 6 (32) or 12 (64); a line's sets of 32 voxels are split evenly over as
// few blocks as that allows (J above 6 is rounded up to an even number).
static int adj_j(int nz, int zrun) {
    const int cap = zrun == 8 ? 2 : zrun == 16 ? 4 : zrun == 32 ? 6 : 12;
    const int sets = (nz + 31) / 32, blocks = (sets + cap - 1) / cap;
    const int J = (sets + blocks - 1) / blocks;
    return J <= 6 ? J : (J + 1) & ~1;
}
// Sets of warps that share a tile's views: by the lines of a frame alone (not by
// the frames, the z-run or the GPU's load, since it groups a voxel's terms).  A^T
// with its step weighting at 24^3 x 4, 32 x 32, 12 views: 37 us with one set, 30
// with two, 26 with four; 40^3 x 4 (100 tiles): 45, 39, 43; 64^3 x 4 (256): 50, 61,
// 69.  A tall volume fills the GPU along z.
static int adj_parts_of_views(const ProjDims& d, int lines_x, int lines_y) {
    const long long tiles = (long long)((lines_x + ADJ_T - 1) / ADJ_T) * ((lines_y + ADJ_T - 1) / ADJ_T);
    return d.nz > 64 ? 1 : tiles <= 64 ? 4 : tiles <= 128 ? 2 : 1;
}
// Columns that a run of ADJ_T lines, str voxels apart, has on the axis, and one more.
static int adj_slots(const ProjDims& d, int str) {
    const double n = ceil((str * (ADJ_T - 1) + 2) * (double)d.vox * d.dsd / d.dso / d.du) + 1.0;
    return n < 2.0 ? 2 : n > 32.0 ? 32 : (int)n;
}
static int adj_nzb(const ProjDims& d, int zrun) {
    const int run = 32 * adj_j(d.nz, zrun);
    return (d.nz + run - 1) / run;
}
static dim3 adj_grid(const ProjDims& d, int zrun) {
    return dim3((d.nx + ADJ_T - 1) / ADJ_T, (d.ny + ADJ_T - 1) / ADJ_T, adj_nzb(d, zrun) * d.nt);
}
template <int MODE>
static void launch_adj_zb(msf_projector* p, const float* e, float* out, const float* a1, float* out2,
                          const CgScalars& cg, float inv_s2, cudaStream_t st) {
    const ProjDims& d = p->dims;
    const int J = adj_j(d.nz, p->adj_zb), slots = adj_slots(d, 1);
    const dim3 grid = adj_grid(d, p->adj_zb);
    const size_t smem = (size_t)ADJ_T * ADJ_T * adj_line(J) * sizeof(float);
#define MSF_ADJ_CASE(N, P)                                                                                          \
    joseph_adj_kernel<MODE, N, P><<<grid, dim3(32, ADJ_T * P), smem * P, st>>>(p->d_col, p->d_trig, p->d_vflag, e, \
                                                                               out, a1, out2, cg, inv_s2, d, slots)
    const int parts = adj_parts_of_views(d, d.nx, d.ny);
    switch (J) {
        case 1: if (parts == 4) MSF_ADJ_CASE(1, 4); else if (parts == 2) MSF_ADJ_CASE(1, 2); else MSF_ADJ_CASE(1, 1); break;
        case 2: if (parts == 4) MSF_ADJ_CASE(2, 4); else if (parts == 2) MSF_ADJ_CASE(2, 2); else MSF_ADJ_CASE(2, 1); break;
        case 3: MSF_ADJ_CASE(3, 1); break;
        case 4: MSF_ADJ_CASE(4, 1); break;
        case 5: MSF_ADJ_CASE(5, 1); break;
        case 6: MSF_ADJ_CASE(6, 1); break;
        case 8: MSF_ADJ_CASE(8, 1); break;
        case 10: MSF_ADJ_CASE(10, 1); break;
        case 12: MSF_ADJ_CASE(12, 1); break;
    }
#undef MSF_ADJ_CASE
}

template <int MODE>
static msf_status launch_adj(msf_projector* p, const float* e, float* out, const float* a1, float* out2,
                             const CgScalars& cg, float inv_s2, cudaStream_t st) {
    MSF_PROF("joseph_adj", st);
    launch_adj_zb<MODE>(p, e, out, a1, out2, cg, inv_s2, st);
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

// Which calls take the planes' kernels (projector_planes.cu), where a warp's 32 lanes are
// detector columns or voxels along x, instead of rows or voxels along z.  The bounds below
// were drawn through times of both on 480 shapes of 16^2 to 512^2 voxels, 1 to 200 slices,
// 1 to 160 rows, 24 to 48 views and 2 to 12 frames (given here as planes' gain over lines).
// Where lanes are spare, the work sets the time once there is enough of it; before that a
// warp's walk does, and the lines' is the shorter.
//   A (the same bits either way): up to a set of 32 rows, from 8000 columns of all frames for
//      one row (128^2 x 1, 85920 columns: 6.7 times) to 34000 for 32 (128^2 x 8, 85920: 1.2;
//      64^2, 42720: 0.95); with two sets, the second of which is short up to 48 rows, by columns
//      x planes (384^2, 51552 columns: 33 rows 1.3 to 1.5, 48 rows 1.0 to 1.1; 48^2, 32160: 0.9).
//   A^T and CG: by the frame alone, since a voxel's terms are grouped otherwise, and a frame
//      must not depend on how many others its problem has (a problem split by time-points
//      equals the whole bit for bit).  The bounds are those of 12 frames, which no number up
//      to that is slower with than the planes; fewer would be faster in lines near them.  Up
//      to 16 slices by the frame's lines of voxels (512^2 x 1 x 2: 3.7 to 7.3 times, 96^2 x 8 x 12:
//      1.4 to 1.7, 96^2 x 16 x 12: 1.0; 96^2 x 8 x 2: 0.50), sooner the more rows a voxel has; above,
//      where the rows are too few for the voxels beside a column (384^2 x 64 x 4, 40 rows: 1.1, 64
//      rows: 0.67), or where CG's slower A outweighs A^T (384^2 x 24 x 4, 33 rows: CG 1.14, A^T 0.97).
//   ICD: its three launches a step tell in favour of lines further (128^2 x 8 x 12: 1.0 to 1.24,
//      96^2 x 8 x 12: 0.76 to 0.96, 256^2 x 16 x 4: 0.87; 384^2 x 16 x 4: 1.18); in a workspace for planes
//      it needs lines of at most 1.5 times the volume, as from eight slices.
static void choose_routes(msf_projector* p) {
    const ProjDims& d = p->dims;
    if (!planes_fit(d)) return;
    const int nz = d.nz, nv = d.nv;
    const double cols = (double)d.nt * d.views * d.nu, xy = (double)d.nx * d.ny;
    p->fwd_planes = nv <= 32 ? cols >= 8000.0 + (nz <= 2 ? 4.0 : 25.0) * nv * nv
                             : nv <= 48 && cols * std::max(d.nx, d.ny) >= 2e6 + 3.3e5 * (nv - 33);
    if (nz <= 16) {
        p->adj_planes = 12.0 * xy >= (16000.0 + 4500.0 * nz) * (nv >= 8 * nz ? 0.6 : nv >= 2 * nz ? 0.72 : 1.0);
    } else if (nz < 24) {
        p->adj_planes = 12.0 * xy >= 200000.0;
    } else {
        const int few = std::max(28, nz / 2 + (nz <= 64 ? 10 : 0));
        p->adj_planes = (nv < few && xy >= (nz <= 64 ? 50000.0 : 32500.0)) ||
                        (3 * nv < 2 * few && xy >= (nz <= 64 ? 12500.0 : 3000.0)) ||
                        (nv <= 48 && xy >= 100000.0 && (nz < 32 || (nz <= 40 && nv < 40)));
    }
    p->icd_planes = p->adj_planes && (nz < 8 || nv < 8 || 2 * nv <= nz || 12.0 * xy >= 18000.0 * nz);
}

static dim3 icd_grid(const ProjDims& d, int gx, int gy, int zrun) {
    const int pairs = (d.nz + 1) / 2, run = 32 * adj_j(pairs, zrun);
    return dim3((gx + ADJ_T - 1) / ADJ_T, (gy + ADJ_T - 1) / ADJ_T, (pairs + run - 1) / run * d.nt);
}

static msf_status launch_icd_group(msf_projector* p, const float* e, const float* z, const float* v,
                                   const float* theta2, float* dlt, IcdSums* S, float inv_s2, const IcdGroup& G,
                                   cudaStream_t st) {
    const ProjDims& d = p->dims;
    const int J = adj_j((d.nz + 1) / 2, p->adj_zb), slots = adj_slots(d, 2);
    const dim3 grid = icd_grid(d, G.gx, G.gy, p->adj_zb);
    const size_t smem = (size_t)ADJ_T * ADJ_T * adj_line(J) * sizeof(float);
    S->gblocks = grid.x * grid.y * (grid.z / d.nt);
    MSF_PROF("icd_group", st);
#define MSF_ICD_CASE(N, P)                                                                                          \
    icd_group_kernel<N, P><<<grid, dim3(32, ADJ_T * P), smem * P, st>>>(p->d_col, p->d_trig, p->d_vflag, e, z, v,  \
                                                                        theta2, dlt, *S, inv_s2, G, d, slots)
    const int parts = adj_parts_of_views(d, par_count(d.nx, 0), par_count(d.ny, 0));
    switch (J) {
        case 1: if (parts == 4) MSF_ICD_CASE(1, 4); else if (parts == 2) MSF_ICD_CASE(1, 2); else MSF_ICD_CASE(1, 1); break;
        case 2: MSF_ICD_CASE(2, 1); break;
        case 3: MSF_ICD_CASE(3, 1); break;
        case 4: MSF_ICD_CASE(4, 1); break;
        case 5: MSF_ICD_CASE(5, 1); break;
        case 6: MSF_ICD_CASE(6, 1); break;
        case 8: MSF_ICD_CASE(8, 1); break;
        case 10: MSF_ICD_CASE(10, 1); break;
        case 12: MSF_ICD_CASE(12, 1); break;
    }
#undef MSF_ICD_CASE
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

}  // namespace msf

using namespace msf;

const msf_vol* msf::projector_volume(const msf_projector* p) { return &p->vol; }
int* msf::dataprox_status(msf_dataprox* d) { return d->d_status; }
size_t msf::projector_sino_size(const msf_projector* p) { return sino_size(p); }
void msf::projector_detector(const msf_projector* p, int* nu, int* nv) {
    *nu = p->geom.nu;
    *nv = p->geom.nv;
}

extern "C" msf_status msf_projector_create(const msf_geom* geom, const msf_vol* vol,
                                           msf_projector** out) {
    MSF_REQUIRE(geom && vol && out, "msf_projector_create: NULL argument");
    *out = nullptr;
    MSF_REQUIRE(vol->nx > 0 && vol->ny > 0 && vol->nz > 0 && vol->nt > 0 && vol->voxel > 0,
                "msf_projector_create: volume sizes and voxel must be positive");
    MSF_REQUIRE(geom->nu > 0 && geom->nv > 0 && geom->views > 0 && geom->du > 0 && geom->dv > 0,
                "msf_projector_create: detector sizes, pitch and views must be positive");
    MSF_REQUIRE(geom->angles != nullptr, "msf_projector_create: angles is NULL");
    const double R = 0.5 * vol->voxel * sqrt((double)vol->nx * vol->nx + (double)vol->ny * vol->ny);
    MSF_REQUIRE(geom->dso > R && geom->dsd - geom->dso > R,
                "msf_projector_create: source (dso=%g) and detector (dsd-dso=%g) must lie outside "
                "the volume's circumscribed cylinder (radius %g)", geom->dso, geom->dsd - geom->dso, R);
    const double vmax = 0.5 * (geom->nv - 1) * geom->dv;
    MSF_REQUIRE(vmax < geom->dsd / sqrt(2.0),
                "msf_projector_create: cone too wide (z-major rays are not modelled)");
    MSF_REQUIRE((size_t)vol->nt * vol->nx * vol->ny * vol->nz < (size_t)1 << 40,
                "msf_projector_create: volume too large");
    MSF_TRY(check_device());

    msf_projector* p = new msf_projector();
    p->geom = *geom;
    p->vol = *vol;
    const int G = vol->nt * geom->views;
    p->angles.assign(geom->angles, geom->angles + G);
    p->geom.angles = p->angles.data();
    ProjDims& d = p->dims;
    d.nx = vol->nx; d.ny = vol->ny; d.nz = vol->nz; d.nt = vol->nt;
    d.nu = geom->nu; d.nv = geom->nv; d.views = geom->views;
    d.cx = 0.5f * (vol->nx - 1); d.cy = 0.5f * (vol->ny - 1); d.cz = 0.5f * (vol->nz - 1);
    d.cu = 0.5f * (geom->nu - 1); d.cv = 0.5f * (geom->nv - 1);
    d.vox = (float)vol->voxel; d.du = (float)geom->du; d.dv = (float)geom->dv;
    d.dso = (float)geom->dso; d.dsd = (float)geom->dsd;

    choose_routes(p);
    const bool planes = p->fwd_planes || p->adj_planes, lines = !p->fwd_planes || !p->adj_planes || !p->icd_planes;
    if (p->adj_planes) p->adj_zb = 16;

    auto cleanup = [&](msf_status st) { msf_projector_destroy(p); return st; };
    const size_t col_bytes = (size_t)G * geom->nu * 2 * sizeof(float4);
    const size_t line_bytes = (VZ_FRONT + vz_pitch(vol->nz)) * sizeof(float);
    const size_t pair_bytes = planes ? vol_size(*vol) * 2 * sizeof(float2) : 0;
    const size_t vz_bytes = lines ? vz_size(*vol) * sizeof(float) : 0;
    const size_t in_bytes = std::max(pair_bytes, (p->adj_planes && !p->icd_planes ? 2 : 1) * vz_bytes);   // ICD: z and v
    const size_t sw_bytes = (p->adj_planes ? sino_size(p) : rows_size(p)) * sizeof(float);
    if (cudaMalloc(&p->d_angles, G * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&p->d_col, col_bytes) != cudaSuccess ||
        cudaMalloc(&p->d_trig, G * sizeof(float2)) != cudaSuccess ||
        cudaMalloc(&p->d_vflag, G * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&p->d_in, in_bytes) != cudaSuccess || cudaMalloc(&p->d_zero, line_bytes) != cudaSuccess ||
        cudaMalloc(&p->d_sw, sw_bytes) != cudaSuccess) {
        cudaGetLastError();
        return cleanup(fail(MSF_ERR_NOMEM, "msf_projector_create: out of device memory"));
    }
    if (lines) p->d_vz = static_cast<float*>(p->d_in);
    if (planes) {
        p->d_px = static_cast<float2*>(p->d_in);
        p->d_py = p->d_px + vol_size(*vol);
    }
    p->bytes = G * sizeof(double) + col_bytes + G * (sizeof(float2) + sizeof(int)) + in_bytes + line_bytes + sw_bytes;
    std::vector<float2> trig(G);
    for (int g = 0; g < G; ++g) trig[g] = make_float2((float)cos(p->angles[g]), (float)sin(p->angles[g]));
    int* d_bad = nullptr;
    int h_bad = 0;
    cudaError_t e = cudaMemcpy(p->d_angles, p->angles.data(), G * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(p->d_trig, trig.data(), G * sizeof(float2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(p->d_vflag, 0, G * sizeof(int));
    if (e == cudaSuccess && lines && !planes) e = cudaMemset(p->d_vz, 0, vz_bytes);   // the lines' margins
    if (e == cudaSuccess) e = cudaMemset(p->d_zero, 0, line_bytes);
    if (e == cudaSuccess) e = cudaMemset(p->d_sw, 0, sw_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&d_bad, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(d_bad, 0, sizeof(int));
    if (e == cudaSuccess) {
        column_table_kernel<<<dim3((geom->nu + 127) / 128, G), 128>>>(p->d_angles, p->d_col, p->d_vflag, d_bad, d, vol->voxel,
                                                                    geom->du, geom->dso, geom->dsd);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h_bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost);
    if (d_bad) cudaFree(d_bad);
    if (e != cudaSuccess) return cleanup(fail(MSF_ERR_CUDA, "msf_projector_create: %s", cudaGetErrorString(e)));
    if (h_bad) return cleanup(fail(MSF_ERR_ARG, "msf_projector_create: a ray's voxel planes are not all "
                                               "between its source and detector"));
    *out = p;
    return MSF_OK;
}

extern "C" void msf_projector_destroy(msf_projector* p) {
    if (!p) return;
    cudaFree(p->d_angles);
    cudaFree(p->d_col);
    cudaFree(p->d_trig);
    cudaFree(p->d_vflag);
    cudaFree(p->d_in);
    cudaFree(p->d_zero);
    cudaFree(p->d_sw);
    delete p;
}

extern "C" size_t msf_projector_bytes(const msf_projector* p) { return p ? p->bytes : 0; }

extern "C" msf_status msf_project(msf_projector* p, const float* d_x, float* d_y, void* stream) {
    MSF_REQUIRE(p && d_x && d_y, "msf_project: NULL argument");
    if (p->fwd_planes) return planes_project(p, d_x, d_y, as_stream(stream));
    return launch_fwd<FWD_PLAIN, false>(p, d_x, d_y, nullptr, nullptr, as_stream(stream));
}

extern "C" msf_status msf_backproject(msf_projector* p, const float* d_y, float* d_x, void* stream) {
    MSF_REQUIRE(p && d_x && d_y, "msf_backproject: NULL argument");
    cudaStream_t st = as_stream(stream);
    if (p->adj_planes) return planes_backproject(p, d_y, d_x, st);
    {
        const ProjDims& d = p->dims;
        MSF_PROF("step_weight", st);
        step_weight_kernel<<<dim3(d.nt * d.views, (d.nu + 31) / 32, (d.nv + 31) / 32), dim3(32, 8), 0, st>>>(
            p->d_col, d_y, p->d_sw, d);
        MSF_LAUNCH_CHECK();
    }
    return launch_adj<ADJ_PLAIN>(p, p->d_sw, d_x, nullptr, nullptr, CgScalars{}, 0.0f, st);
}

// Partial sums of the ICD agent in lines: the largest grids of any group (parity 0) and tuning.
static size_t icd_ipart(const msf_projector* p) {
    const dim3 g = icd_grid(p->dims, par_count(p->vol.nx, 0), par_count(p->vol.ny, 0), 8);
    return (size_t)g.x * g.y * g.z * 2;
}
static size_t icd_spart(const msf_projector* p) {
    return (size_t)((p->dims.nu + 1) / 2) * p->dims.views * fwd_chunks(p->dims) * p->vol.nt;
}

// The data agents' workspace in lines.
static msf_status lines_alloc(msf_dataprox* d) {
    const msf_projector* p = d->p;
    const size_t nl = vz_size(p->vol), nr = rows_size(p);
    const int nt = p->vol.nt;
    const dim3 ga = adj_grid(p->dims, 8);             // the largest block count of any z-run
    const int parts_adj = ga.x * ga.y * adj_nzb(p->dims, 8);
    // blocks of a frame of the vector kernels: eight warps of one line or more each
    const size_t lines = (size_t)p->vol.nx * p->vol.ny;
    d->parts_upd = lines < 8 * 512 ? (int)((lines + 7) / 8) : 512;
    const int parts_max = parts_adj > d->parts_upd ? parts_adj : d->parts_upd;
    if (cudaMalloc(&d->d_rows, nr * 4) != cudaSuccess || cudaMalloc(&d->d_rows2, nr * 4) != cudaSuccess ||
        cudaMalloc(&d->d_ipart, icd_ipart(p) * 8) != cudaSuccess ||
        cudaMalloc(&d->d_spart, icd_spart(p) * 8) != cudaSuccess || cudaMalloc(&d->d_r, nl * 4) != cudaSuccess ||
        cudaMalloc(&d->d_p, nl * 4) != cudaSuccess || cudaMalloc(&d->d_q, nl * 4) != cudaSuccess ||
        cudaMalloc(&d->d_partial, (size_t)nt * parts_max * 8) != cudaSuccess)
        return MSF_ERR_NOMEM;
    d->i_v = d->d_q;
    d->i_theta2 = d->d_r;
    d->i_delta = d->d_p;
    return MSF_OK;
}

// The lines that a projection or a gather reads need their margins cleared; those of d_r
// and d_q are loaded in units of four values at most, and dropped.
static bool lines_clear(msf_dataprox* d) {
    const size_t nl = vz_size(d->p->vol), nr = rows_size(d->p);
    return cudaMemset(d->d_p, 0, nl * 4) == cudaSuccess && cudaMemset(d->d_rows, 0, nr * 4) == cudaSuccess &&
           cudaMemset(d->d_rows2, 0, nr * 4) == cudaSuccess;
}

// The workspace of a plan whose CG takes planes, with the ICD agent's lines in it.
static msf_status planes_alloc(msf_dataprox* d) {
    const msf_projector* p = d->p;
    if (p->icd_planes) return planes_dataprox_alloc(d, 0, 0, 0);
    MSF_TRY(planes_dataprox_alloc(d, rows_size(p), icd_ipart(p), icd_spart(p)));
    d->i_v = p->d_vz + vz_size(p->vol);
    d->i_theta2 = d->d_r;
    d->i_delta = d->d_r + vz_size(p->vol);
    return MSF_OK;
}

extern "C" msf_status msf_dataprox_create(msf_projector* p, msf_dataprox** out) {
    MSF_REQUIRE(p && out, "msf_dataprox_create: NULL argument");
    *out = nullptr;
    msf_dataprox* d = new msf_dataprox();
    d->p = p;
    const int nt = p->vol.nt;
    msf_status st = p->adj_planes ? planes_alloc(d) : lines_alloc(d);
    if (st == MSF_OK &&
        (cudaMalloc(&d->d_count, nt * sizeof(unsigned)) != cudaSuccess || cudaMalloc(&d->d_rr, nt * 8) != cudaSuccess ||
         cudaMalloc(&d->d_alpha, nt * 8) != cudaSuccess || cudaMalloc(&d->d_beta, nt * 8) != cudaSuccess ||
         cudaMalloc(&d->d_status, sizeof(int)) != cudaSuccess))
        st = MSF_ERR_NOMEM;
    if (st != MSF_OK) {
        cudaGetLastError();
        msf_dataprox_destroy(d);
        return fail(st, "msf_dataprox_create: out of device memory");
    }
    if ((!p->adj_planes && !lines_clear(d)) || cudaMemset(d->d_status, 0, sizeof(int)) != cudaSuccess ||
        cudaMemset(d->d_count, 0, nt * sizeof(unsigned)) != cudaSuccess) {
        msf_dataprox_destroy(d);
        return fail(MSF_ERR_CUDA, "msf_dataprox_create: memset failed");
    }
    st = settle_default_stream();
    if (st != MSF_OK) {
        msf_dataprox_destroy(d);
        return st;
    }
    *out = d;
    return MSF_OK;
}

extern "C" void msf_dataprox_destroy(msf_dataprox* d) {
    if (!d) return;
    cudaFree(d->d_r);
    if (!d->d_p2) {   // (planes: one allocation)
        cudaFree(d->d_p);
        cudaFree(d->d_q);
    }
    cudaFree(d->d_count);
    cudaFree(d->d_partial); cudaFree(d->d_rr); cudaFree(d->d_alpha); cudaFree(d->d_beta);
    cudaFree(d->d_status);
    cudaFree(d->d_rows); cudaFree(d->d_rows2); cudaFree(d->d_ipart); cudaFree(d->d_spart);
    delete d;
}

extern "C" msf_status msf_prox_data(msf_dataprox* dp, const float* d_y, const float* d_lambda,
                                    const float* d_v, float* d_x, double sigma, int n_cg, void* stream) {
    MSF_REQUIRE(dp && d_y && d_lambda && d_v && d_x, "msf_prox_data: NULL argument");
    MSF_REQUIRE(sigma > 0 && isfinite(sigma), "msf_prox_data: sigma must be positive");
    MSF_REQUIRE(n_cg >= 0, "msf_prox_data: n_cg must be >= 0");
    if (n_cg == 0) return MSF_OK;
    msf_projector* p = dp->p;
    cudaStream_t st = as_stream(stream);
    const float inv_s2 = (float)(1.0 / (sigma * sigma));
    if (p->adj_planes) return planes_prox_cg(dp, d_y, d_lambda, d_v, d_x, inv_s2, n_cg, st);
    const msf_vol& v = p->vol;
    const size_t lines = (size_t)v.nx * v.ny;
    const dim3 ugrid(dp->parts_upd, v.nt);
    const CgScalars ca{dp->d_partial, dp->d_rr, dp->d_alpha, dp->d_status, dp->d_count};
    const CgScalars cb{dp->d_partial, dp->d_rr, dp->d_beta, dp->d_status, dp->d_count};
    float* z = p->d_vz;
    {   // z and v - z as lines
        MSF_PROF("transpose", st);
        lines_kernel<LINES_PAIR><<<lines_grid(v), 256, 0, st>>>(d_x, z, d_v, dp->d_q, v.nx, v.ny, v.nz, shared_input(p));
        MSF_LAUNCH_CHECK();
    }
    // r = A^T Lambda (y - A z) + (v - z)/sigma^2 ; p = r ; rr = r.r
    MSF_TRY((launch_fwd_lines<FWD_RESIDUAL, true>(p, z, dp->d_rows, d_lambda, d_y, st)));
    MSF_TRY(launch_adj<ADJ_CG_INIT>(p, dp->d_rows, dp->d_r, dp->d_q, dp->d_p, ca, inv_s2, st));
    for (int it = 0; it < n_cg; ++it) {
        // s = Lambda A p ; q = A^T s + p/sigma^2 ; alpha = rr / p.q
        MSF_TRY((launch_fwd_lines<FWD_LAMBDA, true>(p, dp->d_p, dp->d_rows, d_lambda, nullptr, st)));
        MSF_TRY(launch_adj<ADJ_CG_Q>(p, dp->d_rows, dp->d_q, dp->d_p, nullptr, ca, inv_s2, st));
        if (it + 1 == n_cg) break;
        {   // r -= alpha q ; beta = r.r / rr
            MSF_PROF("cg_residual", st);
            cg_residual_kernel<<<ugrid, 256, 0, st>>>(dp->d_r, dp->d_q, dp->d_alpha, cb, lines, v.nz);
            MSF_LAUNCH_CHECK();
        }
        {   // z += alpha p ; p = r + beta p
            MSF_PROF("cg_direction", st);
            cg_direction_kernel<<<ugrid, 256, 0, st>>>(z, dp->d_p, dp->d_r, dp->d_alpha, dp->d_beta, lines, v.nz);
            MSF_LAUNCH_CHECK();
        }
    }
    // the last step's z + alpha p, back in volume order
    MSF_PROF("volume", st);
    volume_kernel<true><<<lines_grid(v), 256, 0, st>>>(z, dp->d_p, dp->d_r, dp->d_q, dp->d_alpha, d_x, dp->d_status, v.nx,
                                                       v.ny, v.nz);
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

extern "C" msf_status msf_prox_data_icd(msf_dataprox* dp, const float* d_y, const float* d_lambda,
                                        const float* d_v, float* d_x, double sigma, int n_sweeps, void* stream) {
    MSF_REQUIRE(dp && d_y && d_lambda && d_v && d_x, "msf_prox_data_icd: NULL argument");
    MSF_REQUIRE(sigma > 0 && isfinite(sigma), "msf_prox_data_icd: sigma must be positive");
    MSF_REQUIRE(n_sweeps >= 0, "msf_prox_data_icd: n_sweeps must be >= 0");
    if (n_sweeps == 0) return MSF_OK;
    msf_projector* p = dp->p;
    cudaStream_t st = as_stream(stream);
    if (p->icd_planes) return planes_prox_icd(dp, d_y, d_lambda, d_v, d_x, sigma, n_sweeps, st);
    const ProjDims& d = p->dims;
    const msf_vol& v = p->vol;
    const int nt = v.nt;
    const float inv_s2 = (float)(1.0 / (sigma * sigma));
    float *z = p->d_vz, *vl = dp->i_v, *theta2 = dp->i_theta2, *dlt = dp->i_delta;
    if (p->adj_planes) {   // the margins, in a workspace that CG overwrites
        MSF_TRY_CUDA(cudaMemsetAsync(dlt, 0, vz_size(v) * sizeof(float), st));
        MSF_TRY_CUDA(cudaMemsetAsync(dp->d_rows, 0, rows_size(p) * sizeof(float), st));
        MSF_TRY_CUDA(cudaMemsetAsync(dp->d_rows2, 0, rows_size(p) * sizeof(float), st));
    }
    {   // z and v as lines
        MSF_PROF("transpose", st);
        lines_kernel<LINES_BOTH><<<lines_grid(v), 256, 0, st>>>(d_x, z, d_v, vl, v.nx, v.ny, v.nz, shared_input(p));
        MSF_LAUNCH_CHECK();
    }
    // e' = step Lambda (y - A z)
    MSF_TRY((launch_fwd_lines<FWD_RESIDUAL, true>(p, z, dp->d_rows, d_lambda, d_y, st)));
    {   // step^2 Lambda, in the buffer that then takes step Lambda (A delta)
        MSF_PROF("icd_weights", st);
        icd_weights_kernel<<<dim3(nt * d.views, (d.nu + 31) / 32, (d.nv + 31) / 32), dim3(32, 8), 0, st>>>(
            p->d_col, d_lambda, dp->d_rows2, d);
        MSF_LAUNCH_CHECK();
    }
    // theta2 = (A^T Lambda A)_ss + 1/sigma^2
    MSF_TRY(launch_adj<ADJ_THETA2>(p, dp->d_rows2, theta2, nullptr, nullptr, CgScalars{}, inv_s2, st));
    IcdSums S{dp->d_ipart, dp->d_spart, 0, dp->d_alpha, 1.0 / (sigma * sigma), dp->d_status, dp->d_count};
    for (int sw = 0; sw < n_sweeps; ++sw) {
        for (int grp = 0; grp < 8; ++grp) {
            IcdGroup G;
            G.px = grp & 1; G.py = (grp >> 1) & 1; G.pz = grp >> 2;
            G.gx = par_count(v.nx, G.px); G.gy = par_count(v.ny, G.py); G.gz = par_count(v.nz, G.pz);
            if (G.gx == 0 || G.gy == 0 || G.gz == 0) continue;
            MSF_TRY(launch_icd_group(p, dp->d_rows, z, vl, theta2, dlt, &S, inv_s2, G, st));
            {   // step Lambda (A delta), and alpha
                MSF_PROF("joseph_fwd", st);
                launch_fwd_kernel<FWD_ICD, true, true>(p, dlt, dp->d_rows2, d_lambda, nullptr, G.px, G.py, S, st);
                MSF_LAUNCH_CHECK();
            }
            {   // e' -= alpha step Lambda (A delta) ; z += alpha delta
                MSF_PROF("icd_update", st);
                const size_t lines = std::max((size_t)d.views * d.nu, (size_t)G.gx * G.gy);
                const int half = (int)std::min<size_t>(256, (lines + 7) / 8);
                icd_update_kernel<<<dim3(2 * half, nt), 256, 0, st>>>(dp->d_rows, dp->d_rows2, z, dlt, dp->d_alpha, G, d);
                MSF_LAUNCH_CHECK();
            }
        }
    }
    MSF_PROF("volume", st);
    volume_kernel<false><<<lines_grid(v), 256, 0, st>>>(z, nullptr, nullptr, nullptr, nullptr, d_x, nullptr, v.nx, v.ny, v.nz);
    MSF_LAUNCH_CHECK();
    return MSF_OK;
}

extern "C" msf_status msf_phantom_voxelize(const msf_vol* vol, const double* h_ell, int n_ell, int ss,
                                           float* d_x, void* stream) {
    MSF_REQUIRE(vol && h_ell && d_x, "msf_phantom_voxelize: NULL argument");
    MSF_REQUIRE(n_ell > 0 && ss > 0 && (size_t)n_ell * vol->nt <= MSF_MAX_ELL_RECORDS,
                "msf_phantom_voxelize: need 0 < n_ell*nt <= %d and ss > 0", MSF_MAX_ELL_RECORDS);
    cudaStream_t st = as_stream(stream);
    MSF_TRY_CUDA(cudaMemcpyToSymbolAsync(c_ell, h_ell, (size_t)n_ell * vol->nt * 16 * sizeof(double), 0,
                                         cudaMemcpyHostToDevice, st));
    phantom_voxelize_kernel<<<152 * 8, 256, 0, st>>>(d_x, vol->nx, vol->ny, vol->nz, vol->nt, vol->voxel, n_ell, ss);
    MSF_LAUNCH_CHECK();
    MSF_TRY_CUDA(cudaStreamSynchronize(st));   // c_ell is reused by the next call
    return MSF_OK;
}

extern "C" msf_status msf_phantom_project(msf_projector* p, const double* h_ell, int n_ell, float* d_y,
                                          void* stream) {
    MSF_REQUIRE(p && h_ell && d_y, "msf_phantom_project: NULL argument");
    MSF_REQUIRE(n_ell > 0 && (size_t)n_ell * p->vol.nt <= MSF_MAX_ELL_RECORDS,
                "msf_phantom_project: need 0 < n_ell*nt <= %d", MSF_MAX_ELL_RECORDS);
    cudaStream_t st = as_stream(stream);
    MSF_TRY_CUDA(cudaMemcpyToSymbolAsync(c_ell, h_ell, (size_t)n_ell * p->vol.nt * 16 * sizeof(double), 0,
                                         cudaMemcpyHostToDevice, st));
    phantom_project_kernel<<<152 * 8, 256, 0, st>>>(p->d_angles, d_y, p->dims, p->geom.du, p->geom.dv,
                                                    p->geom.dso, p->geom.dsd, n_ell);
    MSF_LAUNCH_CHECK();
    MSF_TRY_CUDA(cudaStreamSynchronize(st));
    return MSF_OK;
}

// ====================================================================== no-allocation forward projection
//
// msf_project_static: the forward projection of msf_project for callers that
// cannot allocate device memory.  The per-column ray table that a projector
// plan would own lives instead in the file-scope device array below, of fixed
// size, which every GPU that loads this library keeps until the process exits.
// The frame is read in its natural layout for both ray families (no transposed
// copy), so the caller's input and output are the only other memory touched.

namespace msf {

constexpr size_t STATIC_SCRATCH_BYTES = (size_t)8 << 20;   // 8 MiB
constexpr int STATIC_MAX_VIEWS = 8192;                      // nt * views
constexpr size_t STATIC_MAX_COLUMNS = 250000;               // nt * views * nu

static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

// Layout inside the array: [angles: G doubles][column table: G*nu*32 B]
// [view flags: G ints][geometry flag: 1 int].
static_assert(STATIC_MAX_VIEWS * 8 + STATIC_MAX_COLUMNS * 32 + STATIC_MAX_VIEWS * 4 + 256 <= STATIC_SCRATCH_BYTES,
              "static scratch too small for its stated limits");

// Joseph forward projection reading the frame [nz][ny][nx] for both ray
// families.  Per crossing it performs the forward's operations with the same
// explicit roundings (the lerp v00 + w_a (v01 - v00) along a, then along z,
// and a round-to-nearest accumulation over increasing planes), and a plane
// whose taps all lie outside the grid adds exactly zero in joseph_fwd_kernel,
// so the result equals msf_project's bit for bit; only the addressing differs (the
// volume's own order here instead of lines along z or planes of pairs).
__global__ void __launch_bounds__(128) joseph_fwd_direct_kernel(const float* __restrict__ x,
                                                                const float4* __restrict__ col,
                                                                float* __restrict__ out, ProjDims d) {
    const int iu = blockIdx.x * 32 + threadIdx.x;
    const int iv = blockIdx.y * 4 + threadIdx.y;
    const int g = blockIdx.z;
    if (iu >= d.nu || iv >= d.nv) return;
    const int t = g / d.views;
    const ColParams c = load_col(col, (size_t)g * d.nu + iu);
    const bool xmaj = c.xmajor != 0.0f;
    const int nmaj = xmaj ? d.nx : d.ny, na = xmaj ? d.ny : d.nx;
    const float* __restrict__ vol = x + (size_t)t * d.nx * d.ny * d.nz;
    // element (iz, plane k, minor ia): x-major -> x[iz][ia][k], y-major -> x[iz][k][ia]
    const ptrdiff_t s_maj = xmaj ? 1 : d.nx, s_min = xmaj ? d.nx : 1;
    const ptrdiff_t s_z = (ptrdiff_t)d.nx * d.ny;
    const float cmaj = xmaj ? d.cx : d.cy;
    const RayZ rz = ray_z(c, det_v(iv, d), d.cz);
    float acc = 0.0f;
    for (int k = 0; k < nmaj; ++k) {
        const float tk = __fsub_rn((float)k, cmaj);
        const float fa = __fmaf_rn(tk, c.ba, c.fa_mid);
        const float fz = __fmaf_rn(tk, rz.bz, rz.fz_mid);
        const float a0f = floorf(fa), z0f = floorf(fz);
        if (a0f < -1.0f || a0f > (float)(na - 1) || z0f < -1.0f || z0f > (float)(d.nz - 1)) continue;
        const float wa1 = __fsub_rn(fa, a0f), wz1 = __fsub_rn(fz, z0f);
        const int ia = (int)a0f, iz = (int)z0f;
        const bool a_in0 = ia >= 0, a_in1 = ia + 1 < na;
        const bool z_in0 = iz >= 0, z_in1 = iz + 1 < d.nz;
        const float* p00 = vol + iz * s_z + k * s_maj + ia * s_min;
        const float v00 = (z_in0 && a_in0) ? __ldg(p00) : 0.0f;
        const float v01 = (z_in0 && a_in1) ? __ldg(p00 + s_min) : 0.0f;
        const float v10 = (z_in1 && a_in0) ? __ldg(p00 + s_z) : 0.0f;
        const float v11 = (z_in1 && a_in1) ? __ldg(p00 + s_z + s_min) : 0.0f;
        const float top = __fmaf_rn(wa1, __fsub_rn(v01, v00), v00);
        const float bot = __fmaf_rn(wa1, __fsub_rn(v11, v10), v10);
        acc = __fadd_rn(acc, __fmaf_rn(wz1, __fsub_rn(bot, top), top));
    }
    out[((size_t)g * d.nv + iv) * d.nu + iu] = __fmul_rn(acc, rz.step);
}

// Device address of g_static_scratch for each device, looked up once per
// device (with that device current) on the first call made on it.
static std::mutex g_static_mu;
static void* g_static_ptr[128] = {nullptr};

}  // namespace msf

extern "C" msf_status msf_project_static(const msf_geom* geom, const msf_vol* vol, const float* d_x, float* d_y,
                                         void* stream) {
    MSF_REQUIRE(geom && vol && d_x && d_y && geom->angles, "msf_project_static: NULL argument");
    MSF_REQUIRE(vol->nx > 0 && vol->ny > 0 && vol->nz > 0 && vol->nt > 0 && vol->voxel > 0,
                "msf_project_static: volume sizes and voxel must be positive");
    MSF_REQUIRE(geom->nu > 0 && geom->nv > 0 && geom->views > 0 && geom->du > 0 && geom->dv > 0,
                "msf_project_static: detector sizes, pitch and views must be positive");
    const long long G = (long long)vol->nt * geom->views;
    MSF_REQUIRE(G <= STATIC_MAX_VIEWS && (size_t)G * geom->nu <= STATIC_MAX_COLUMNS,
                "msf_project_static: nt*views = %lld and nt*views*nu = %lld exceed the static table "
                "(at most %d views and %zu view-columns); use msf_projector_create + msf_project",
                G, G * geom->nu, STATIC_MAX_VIEWS, STATIC_MAX_COLUMNS);
    const double R = 0.5 * vol->voxel * sqrt((double)vol->nx * vol->nx + (double)vol->ny * vol->ny);
    MSF_REQUIRE(geom->dso > R && geom->dsd - geom->dso > R,
                "msf_project_static: source and detector must lie outside the volume's circumscribed cylinder");
    MSF_REQUIRE(0.5 * (geom->nv - 1) * geom->dv < geom->dsd / sqrt(2.0),
                "msf_project_static: cone too wide (z-major rays are not modelled)");
    // The voxel planes of every ray must lie between its source and detector.
    // This is checked here in FP64 on the host for every (view, column) -- at
    // most STATIC_MAX_COLUMNS evaluations -- with the formulas of
    // column_table_kernel, so no device flag has to be read back (the table
    // kernel still writes its flag into the array; nothing reads it).  Checking
    // only the end columns would not do: where a view's columns switch between
    // x-major and y-major, the first column of the inner segment can fail alone.
    for (long long g = 0; g < G; ++g) {
        const double th = geom->angles[g], c = cos(th), s = sin(th);
        const double sx = geom->dso * c, sy = geom->dso * s;
        for (int iu = 0; iu < geom->nu; ++iu) {
            const double u = (iu - 0.5 * (geom->nu - 1)) * geom->du;
            const double dx = -(geom->dsd - geom->dso) * c - u * s - sx, dy = -(geom->dsd - geom->dso) * s + u * c - sy;
            const bool xm = fabs(dx) >= fabs(dy);
            const double dmaj = xm ? dx : dy, smaj = xm ? sx : sy;
            const int nmaj = xm ? vol->nx : vol->ny;
            const double l1 = (-0.5 * (nmaj - 1) * vol->voxel - smaj) / dmaj;
            const double l2 = (0.5 * (nmaj - 1) * vol->voxel - smaj) / dmaj;
            MSF_REQUIRE(fmin(l1, l2) > 0.0 && fmax(l1, l2) < 1.0,
                        "msf_project_static: a ray's voxel planes are not all between its source and detector "
                        "(view %lld, column %d)", g, iu);
        }
    }
    int dev = 0;
    MSF_TRY_CUDA(cudaGetDevice(&dev));
    MSF_REQUIRE(dev >= 0 && dev < 128, "msf_project_static: device index %d out of range", dev);
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_static_mu);
        if (!g_static_ptr[dev]) {
            MSF_TRY(check_device());
            cudaError_t e = cudaGetSymbolAddress(&g_static_ptr[dev], g_static_scratch);
            if (e != cudaSuccess) {
                g_static_ptr[dev] = nullptr;
                return fail(MSF_ERR_CUDA, "msf_project_static: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            }
        }
        base = g_static_ptr[dev];
    }
    unsigned char* b = static_cast<unsigned char*>(base);
    double* d_angles = reinterpret_cast<double*>(b);
    float4* d_col = reinterpret_cast<float4*>(b + (size_t)STATIC_MAX_VIEWS * 8);
    int* d_vflag = reinterpret_cast<int*>(b + (size_t)STATIC_MAX_VIEWS * 8 + STATIC_MAX_COLUMNS * 32);
    int* d_bad = d_vflag + STATIC_MAX_VIEWS;
    ProjDims d;
    d.nx = vol->nx; d.ny = vol->ny; d.nz = vol->nz; d.nt = vol->nt;
    d.nu = geom->nu; d.nv = geom->nv; d.views = geom->views;
    d.cx = 0.5f * (vol->nx - 1); d.cy = 0.5f * (vol->ny - 1); d.cz = 0.5f * (vol->nz - 1);
    d.cu = 0.5f * (geom->nu - 1); d.cv = 0.5f * (geom->nv - 1);
    d.vox = (float)vol->voxel; d.du = (float)geom->du; d.dv = (float)geom->dv;
    d.dso = (float)geom->dso; d.dsd = (float)geom->dsd;
    cudaStream_t st = as_stream(stream);
    // the array keeps the previous call's contents: the flags start at zero
    MSF_TRY_CUDA(cudaMemcpyAsync(d_angles, geom->angles, G * sizeof(double), cudaMemcpyHostToDevice, st));
    MSF_TRY_CUDA(cudaMemsetAsync(d_vflag, 0, G * sizeof(int), st));
    MSF_TRY_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int), st));
    {
        MSF_PROF("column_table", st);
        column_table_kernel<<<dim3((geom->nu + 127) / 128, (unsigned)G), 128, 0, st>>>(
            d_angles, d_col, d_vflag, d_bad, d, vol->voxel, geom->du, geom->dso, geom->dsd);
        MSF_LAUNCH_CHECK();
    }
    {
        MSF_PROF("joseph_fwd_direct", st);
        joseph_fwd_direct_kernel<<<dim3((d.nu + 31) / 32, (d.nv + 3) / 4, (unsigned)G), dim3(32, 4), 0, st>>>(
            d_x, d_col, d_y, d);
        MSF_LAUNCH_CHECK();
    }
    return MSF_OK;
}

// ====================================================================== autotuning

namespace msf {
uint64_t projector_tuning_gen(const msf_projector* p) { return p ? p->tuning_gen : 0; }
}  // namespace msf

extern "C" msf_status msf_projector_set_tuning(msf_projector* p, int fwd_cols, int fwd_rows, int adj_zrun) {
    MSF_REQUIRE(p, "msf_projector_set_tuning: NULL plan");
    MSF_REQUIRE((fwd_cols == 32 && fwd_rows == 4) || (fwd_cols == 64 && fwd_rows == 2) ||
                    (fwd_cols == 16 && fwd_rows == 8),
                "msf_projector_set_tuning: forward block %dx%d is not 32x4, 64x2 or 16x8", fwd_cols, fwd_rows);
    MSF_REQUIRE(adj_zrun == 8 || adj_zrun == 16 || adj_zrun == 32 || adj_zrun == 64,
                "msf_projector_set_tuning: adjoint z-run %d is not 8, 16, 32 or 64", adj_zrun);
    p->fwd_bx = fwd_cols;
    p->fwd_by = fwd_rows;
    p->adj_zb = adj_zrun;
    ++p->tuning_gen;
    return MSF_OK;
}

extern "C" msf_status msf_projector_autotune(msf_projector* p, void* stream, int* h_choice) {
    MSF_REQUIRE(p, "msf_projector_autotune: NULL plan");
    cudaStream_t st = as_stream(stream);
    const size_t nv = vol_size(p->vol), ns = sino_size(p);
    // inputs: the plan's own scratch, whose values the timing does not depend on (pairs and
    // step-weighted sinogram are cleared); outputs go to a temporary buffer allocated here
    float* tmp = nullptr;
    MSF_TRY_CUDA(cudaMalloc(&tmp, (nv > ns ? nv : ns) * sizeof(float)));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    msf_status st_ = MSF_OK;
    auto time_it = [&](auto&& fn) -> float {
        fn();   // warm
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) fn();
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    MSF_TRY_CUDA(cudaMemsetAsync(p->d_sw, 0, (p->adj_planes ? sino_size(p) : rows_size(p)) * sizeof(float), st));
    if (p->d_px) MSF_TRY_CUDA(cudaMemsetAsync(p->d_px, 0, 2 * nv * sizeof(float2), st));
    const int shapes[3][2] = {{32, 4}, {64, 2}, {16, 8}};
    float best = 1e30f;
    int bi = 0;
    for (int i = 0; i < 3; ++i) {
        p->fwd_bx = shapes[i][0];
        p->fwd_by = shapes[i][1];
        const float ms = time_it([&] {   // A's kernel, and the agents' where they take the other layout
            if (p->fwd_planes || p->adj_planes) planes_project_pairs(p, tmp, st);
            if (!p->fwd_planes || !p->adj_planes)
                launch_fwd_kernel<FWD_PLAIN, false, false>(p, p->d_vz, tmp, nullptr, nullptr, 0, 0, IcdSums{}, st);
        });
        if (ms < best) { best = ms; bi = i; }
    }
    p->fwd_bx = shapes[bi][0];
    p->fwd_by = shapes[bi][1];
    // Planes: z-runs of 64 halve the gather's block count; they are tried only while their grid
    // stays at least 24 waves deep (8 blocks per SM), because with a shallower grid, run beside
    // other problems' kernels (a batch), the longer blocks measured slower although they won when
    // timed alone.  Lines: a run that gives a block the same voxels as one already timed is the
    // same launch; otherwise what wins alone wins beside others, in shallow grids too (CG of
    // 256^3 x 4 with runs of 32 and 64: 10.95 and 10.31 ms, four at once 42.0 and 39.4; 64^2 x 224 x 2,
    // 512 blocks: 0.560 and 0.505, eight at once 3.07 and 2.94).
    const int zbs[4] = {8, 16, 32, 64};
    int nsm = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        nsm = 0;
    const bool deep64 = nsm > 0 && (double)planes_adj_blocks(p->dims, 64) * p->dims.nt >= 24.0 * 8.0 * nsm;
    best = 1e30f;
    int bz = 0;
    for (int i = 0; i < 4; ++i) {
        if (p->adj_planes ? i == 3 && !deep64 : i > 0 && adj_j(p->dims.nz, zbs[i]) == adj_j(p->dims.nz, zbs[i - 1])) continue;
        p->adj_zb = zbs[i];
        const float ms = time_it([&] {
            if (p->adj_planes) planes_gather(p, p->d_sw, tmp, st);
            else launch_adj_zb<ADJ_PLAIN>(p, p->d_sw, tmp, nullptr, nullptr, CgScalars{}, 0.0f, st);
        });
        if (ms < best) { best = ms; bz = i; }
    }
    p->adj_zb = zbs[bz];
    ++p->tuning_gen;
    if (cudaGetLastError() != cudaSuccess) st_ = fail(MSF_ERR_CUDA, "msf_projector_autotune: a trial launch failed");
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(tmp);
    if (h_choice) {
        h_choice[0] = p->fwd_bx;
        h_choice[1] = p->fwd_by;
        h_choice[2] = p->adj_zb;
    }
    return st_;
}
