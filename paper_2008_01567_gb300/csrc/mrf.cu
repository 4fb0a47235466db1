// 4D q-GGMRF prior proximal map (Sec. III, Eq. (5) with the 4D MRF prior of
// Sec. VII: 26 spatial + 2 temporal neighbours) by 16-colour ICD, and the
// direct MAP solve of Eq. (3) with that prior (the MBIR + 4D-MRF comparison of
// Sec. VI) by majorise-minimise with CG on the surrogate problem.
//
// The 16 parity colours ((pt*2+pz)*2+py)*2+px never contain two neighbours,
// so all voxels of one colour update in parallel and the sweep is
// deterministic: the GPU reproduces a sequential colour-ordered sweep exactly
// in real arithmetic.  One launch per colour.
#include <math.h>

#include "common.cuh"

namespace msf {

// Scale of the terms 1 + r whose product shares a reciprocal (qggmrf_pair).
constexpr float MRF_SCALE = 0x1p-33f;
enum MrfKind { MRF_USUAL = 0, MRF_NEAR = 1, MRF_APART = 2 };   // of arithmetic (qggmrf_pair)

struct MrfDims {
    int nx, ny, nz, nt;
    int px, py, pz, pt;          // parities of the colour
    int hx, hy, hz, ht;          // voxels of that colour along each axis
    float inv_s2;                // 1/sigma^2
    float inv_tsx;               // 1/(T sigma_x)
    float pq;                    // p - q
    // surrogate coefficients of the face, edge, corner and temporal neighbours,
    // 2 b a(D) = w (k1 + k2 w) with w = 1 / (1 + r): 2 b (q/p) / (2 sigma_x^2) and
    // 2 b (1 - q/p) / (2 sigma_x^2)  (p = 2); MRF_USUAL: w is 1 / MRF_SCALE times that, and k1 and
    // k2 MRF_SCALE and its square times
    float k1[4], k2[4];
    int kind;
    float bt;                    // temporal weight
};

__device__ __forceinline__ float lg2_ftz(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float lg2_full(float x) {   // of subnormal numbers too
    float r;
    asm("lg2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_ftz(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Twice the weighted surrogate coefficients b a(D) of two neighbours of one kind
// (packed), a(D) = rho'(D)/(2D) of the q-GGMRF potential with p = 2:
//   a(D) = 1/(2 sx^2) * (1 + (q/p) r)/(1 + r)^2,   r = |D/(T sx)|^(p-q),
// in partial fractions of 1/(1 + r).  r is formed as exp2((p-q) log2 .) with the
// hardware approximations (about 2^-21 relative, far inside the FP32 tolerance of
// the agent).  The two share a reciprocal, since the special function unit bounds these
// kernels (28 neighbours, a logarithm, a power and a reciprocal each).
//   MRF_USUAL: p - q >= 0.2.  A ratio below 2^-126 is flushed to r = 0: its r is below
//     2^-25, and the sum 1 either way.  The terms are formed MRF_SCALE times as large, so
//     that their product stays a normal number for any FP32 r beside one of 2^64: unscaled
//     it passed 2^126 at two outliers of 2^63, and both weights vanished, though with q = 1
//     an outlier's influence does not fall with its distance.
//   MRF_NEAR: p - q < 0.2.  r is at most 2^26, no product overflows; the logarithm takes
//     subnormal ratios, which the power brings back to the size of the 1.
//   MRF_APART: coefficients that would lose bits to the scale; a reciprocal each.
template <int KIND>
__device__ __forceinline__ f32x2 qggmrf_pair(f32x2 D, int kind, const MrfDims& m) {
    float r0 = 1.0f, r1 = 1.0f;
    if (m.pq != 0.0f) {
        float d0, d1;
        unpack2(mul2(D, pack2(m.inv_tsx, m.inv_tsx)), d0, d1);
        d0 = KIND == MRF_USUAL ? lg2_ftz(fabsf(d0)) : lg2_full(fabsf(d0));
        d1 = KIND == MRF_USUAL ? lg2_ftz(fabsf(d1)) : lg2_full(fabsf(d1));
        unpack2(mul2(pack2(d0, d1), pack2(m.pq, m.pq)), d0, d1);
        r0 = ex2_ftz(d0);
        r1 = ex2_ftz(d1);
    }
    constexpr float S = KIND == MRF_USUAL ? MRF_SCALE : 1.0f;
    float x, y;
    unpack2(fma2(pack2(r0, r1), pack2(S, S), pack2(S, S)), x, y);
    f32x2 w;
    if (KIND != MRF_APART) {
        const float rc = rcp_ftz(__fmul_rn(x, y));
        w = mul2(pack2(y, x), pack2(rc, rc));
    } else {
        w = pack2(rcp_ftz(x), rcp_ftz(y));
    }
    return mul2(w, fma2(w, pack2(m.k2[kind], m.k2[kind]), pack2(m.k1[kind], m.k1[kind])));
}

// Calls f(offset 1, inside 1, offset 2, inside 2, kind) for the 13 pairs of
// opposite spatial neighbours of voxel (ix, iy, iz) of frame t and its temporal
// pair; offsets in elements.  INNER: the voxel has neighbours on both sides of
// every axis but x.
template <bool INNER, typename F>
__device__ __forceinline__ void neighbour_pairs(int ix, int iy, int iz, int t, const MrfDims& m, F&& f) {
    const ptrdiff_t sx = 1, sy = m.nx, sz = (ptrdiff_t)m.nx * m.ny, st = sz * m.nz;
    const bool xl = ix > 0, xh = ix + 1 < m.nx;
    const bool yl = INNER || iy > 0, yh = INNER || iy + 1 < m.ny, zl = INNER || iz > 0, zh = INNER || iz + 1 < m.nz;
    f(-sx, xl, sx, xh, 0);
    f(-sy, yl, sy, yh, 0);
    f(-sz, zl, sz, zh, 0);
    f(-sy - sx, yl && xl, sy + sx, yh && xh, 1);
    f(-sy + sx, yl && xh, sy - sx, yh && xl, 1);
    f(-sz - sx, zl && xl, sz + sx, zh && xh, 1);
    f(-sz + sx, zl && xh, sz - sx, zh && xl, 1);
    f(-sz - sy, zl && yl, sz + sy, zh && yh, 1);
    f(-sz + sy, zl && yh, sz - sy, zh && yl, 1);
    f(-sz - sy - sx, zl && yl && xl, sz + sy + sx, zh && yh && xh, 2);
    f(-sz - sy + sx, zl && yl && xh, sz + sy - sx, zh && yh && xl, 2);
    f(-sz + sy - sx, zl && yh && xl, sz - sy + sx, zh && yl && xh, 2);
    f(-sz + sy + sx, zl && yh && xh, sz - sy - sx, zh && yl && xl, 2);
    f(-st, INNER || t > 0, st, INNER || t + 1 < m.nt, 3);
}

__device__ __forceinline__ bool inner(int iy, int iz, int t, const MrfDims& m) {
    return iy > 0 && iy + 1 < m.ny && iz > 0 && iz + 1 < m.nz && t > 0 && t + 1 < m.nt;
}

// The minimiser of voxel (ix, iy, iz) of frame t given its neighbours (v may be z: no
// __restrict__, which would let loads of v miss the last sweep's values).
template <int KIND>
__device__ __forceinline__ void icd_voxel(const float* v, float* z, int ix, int iy, int iz,
                                          int t, const MrfDims& m) {
    float* c = z + (((size_t)t * m.nz + iz) * m.ny + iy) * m.nx + ix;
    const float zs = *c;
    f32x2 num = pack2(v[c - z] * m.inv_s2, 0.0f), den = pack2(m.inv_s2, 0.0f);
    auto pair = [&](ptrdiff_t o1, bool in1, ptrdiff_t o2, bool in2, int kind) {
        const f32x2 zr = pack2(in1 ? c[o1] : zs, in2 ? c[o2] : zs);
        float a1, a2;
        unpack2(qggmrf_pair<KIND>(sub2(pack2(zs, zs), zr), kind, m), a1, a2);
        const f32x2 a = pack2(in1 ? a1 : 0.0f, in2 ? a2 : 0.0f);
        num = fma2(a, zr, num);
        den = add2(den, a);
    };
    // (a warp of icd_colour_kernel has one y, z and t)
    if (inner(iy, iz, t, m)) neighbour_pairs<true>(ix, iy, iz, t, m, pair);
    else neighbour_pairs<false>(ix, iy, iz, t, m, pair);
    float n0, n1, d0, d1;
    unpack2(num, n0, n1);
    unpack2(den, d0, d1);
    *c = (n0 + n1) / (d0 + d1);
}

// One colour of a sweep.  Bound by the special function unit (70 operations per
// voxel, 16 lanes a clock) and, close behind, by instruction issue: with an IEEE
// division per neighbour, general exp2 / log2 and one sum of all 28 terms, two
// sweeps of 192^3 x 12 took 7.12 ms; with shared reciprocals and partial fractions
// 3.8, packed pairs (which also halve the sums' length: error against FP64 9.9e-8
// -> 7.4e-8) 3.18, without bounds checks in y, z and t inside the volume 3.12, and, with
// the scaled terms, twelve blocks per SM asked for (BLOCKS; 40 registers) 3.07 (3.38 at the
// 48 that the compiler takes by itself, which a colour of few blocks, waiting for one
// voxel's chain, is faster with: 33^3 x 4 131 against 170 us, 64^3 x 4 180 against 197,
// 110^3 x 3 329 against 326).
template <int KIND, int BLOCKS>
__global__ void __launch_bounds__(128, BLOCKS) icd_colour_kernel(const float* __restrict__ v,
                                                         float* __restrict__ z, MrfDims m) {
    const int hxv = blockIdx.x * 32 + threadIdx.x;
    const int hyv = blockIdx.y * 4 + threadIdx.y;
    const int hzv = blockIdx.z % m.hz;
    const int htv = blockIdx.z / m.hz;
    if (hxv >= m.hx || hyv >= m.hy) return;
    icd_voxel<KIND>(v, z, 2 * hxv + m.px, 2 * hyv + m.py, 2 * hzv + m.pz, 2 * htv + m.pt, m);
}

// All sweeps of a small volume in one launch: the CTAs of one cluster (8 SMs) take
// a colour's voxels, one each, and meet at the cluster's barrier between colours.
// Issuing launches sets the time of such a volume, 16 a sweep (66 us; 33 with one frame): so
// 39 us at 8^3 x 2, 29 at 24^3 and 32^3, 53 at 32^3 x 2, 64 at 24^3 x 4, 68 at 16^3 x 16 (the
// largest, 4096 voxels per colour on 8 SMs).  Replayed from a graph sixteen launches cost
// less than the cluster's barriers and few SMs (31 against 39 us at 8^3 x 2, 37 against 64 at
// 24^3 x 4), so a captured call takes them.
constexpr int ICD_CLUSTER = 8, ICD_SMALL_THREADS = 512;
constexpr long long ICD_SMALL_VOXELS = (long long)ICD_CLUSTER * ICD_SMALL_THREADS;   // of the largest colour
template <int KIND>
__global__ void __cluster_dims__(ICD_CLUSTER, 1, 1) __launch_bounds__(ICD_SMALL_THREADS)
    icd_small_kernel(const float* v, float* z, MrfDims m, int n_sweeps) {
    const int id = blockIdx.x * ICD_SMALL_THREADS + threadIdx.x;
    for (int k = 0; k < 16 * n_sweeps; ++k) {
        const int px = k & 1, py = (k >> 1) & 1, pz = (k >> 2) & 1, pt = (k >> 3) & 1;
        const int hx = (m.nx - px + 1) / 2, hy = (m.ny - py + 1) / 2, hz = (m.nz - pz + 1) / 2, ht = (m.nt - pt + 1) / 2;
        if (hx * hy * hz * ht == 0) continue;   // of a volume of one slice or frame, in every CTA
        if (id < hx * hy * hz * ht) {
            const int x = id % hx, r = id / hx, y = r % hy, q = r / hy;
            icd_voxel<KIND>(v, z, 2 * x + px, 2 * y + py, 2 * (q % hz) + pz, 2 * (q / hz) + pt, m);
        }
        // the colour's voxels, written by any CTA, before the next colour reads them
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}

// ------------------------------------------------------------------ direct MAP

constexpr int MAP_BLOCKS = 152 * 8;

// (L_a x)_s = sum_r b_sr a(anchor_s - anchor_r) (x_s - x_r) over the 26 spatial
// and 2 temporal neighbours of s (free boundaries): half the gradient of the
// prior's quadratic surrogate built at `anchor`.
template <int KIND>
__device__ __forceinline__ float surrogate_lap(const float* __restrict__ anchor, const float* __restrict__ x,
                                               size_t s, int ix, int iy, int iz, int t, const MrfDims& m) {
    const float as = anchor[s], xs = x[s];
    f32x2 acc = 0;
    neighbour_pairs<false>(ix, iy, iz, t, m, [&](ptrdiff_t o1, bool in1, ptrdiff_t o2, bool in2, int kind) {
        const f32x2 ar = pack2(in1 ? anchor[s + o1] : as, in2 ? anchor[s + o2] : as);
        const f32x2 xr = pack2(in1 ? x[s + o1] : xs, in2 ? x[s + o2] : xs);   // outside: a zero difference
        acc = fma2(qggmrf_pair<KIND>(sub2(pack2(as, as), ar), kind, m), sub2(pack2(xs, xs), xr), acc);
    });
    float a0, a1;
    unpack2(acc, a0, a1);
    return 0.5f * (a0 + a1);   // the pairs carry twice the coefficients
}

enum MapLapMode { MAP_INIT = 0, MAP_Q = 1 };

// MAP_INIT: r = data - 2 beta L_a x  (data = A^T Lambda (y - A x) held in r),
//           d = r, partial r.r
// MAP_Q:    q = data + 2 beta L_a d  (data = A^T Lambda A d held in q), partial d.q
// One grid-stride pass over all voxels; per-block FP64 partials.
template <int MODE, int KIND>
__global__ void __launch_bounds__(256) map_lap_kernel(const float* __restrict__ anchor, const float* __restrict__ x,
                                                      float* __restrict__ out, float* __restrict__ out2,
                                                      float two_beta, MrfDims m, double* __restrict__ partial) {
    const size_t sxy = (size_t)m.nx * m.ny, fs = sxy * m.nz, N = fs * m.nt;
    double dot = 0.0;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < N; s += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(s / fs);
        const size_t r = s - (size_t)t * fs;
        const int iz = (int)(r / sxy);
        const int rr = (int)(r - (size_t)iz * sxy);
        const int iy = rr / m.nx, ix = rr - iy * m.nx;
        const float L = surrogate_lap<KIND>(anchor, x, s, ix, iy, iz, t, m);
        if (MODE == MAP_INIT) {
            const float v = fmaf(-two_beta, L, out[s]);
            out[s] = v;
            out2[s] = v;
            dot += (double)v * (double)v;
        } else {
            const float v = fmaf(two_beta, L, out[s]);
            out[s] = v;
            dot += (double)x[s] * (double)v;
        }
    }
    const double b = block_sum_f64(dot);
    if (threadIdx.x == 0) partial[blockIdx.x] = b;
}

template <int MODE>
static void launch_map_lap(const float* anchor, const float* x, float* out, float* out2, float two_beta, const MrfDims& m,
                           double* partial, cudaStream_t st) {
    auto* f = m.kind == MRF_USUAL ? map_lap_kernel<MODE, MRF_USUAL>
              : m.kind == MRF_NEAR ? map_lap_kernel<MODE, MRF_NEAR> : map_lap_kernel<MODE, MRF_APART>;
    f<<<MAP_BLOCKS, 256, 0, st>>>(anchor, x, out, out2, two_beta, m, partial);
}

// x += alpha d ; r -= alpha q ; partial r.r
__global__ void __launch_bounds__(256) map_update_kernel(float* __restrict__ x, float* __restrict__ r,
                                                         const float* __restrict__ d, const float* __restrict__ q,
                                                         const double* __restrict__ scal, size_t N,
                                                         double* __restrict__ partial) {
    const float a = (float)scal[1];
    double dot = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        x[i] = fmaf(a, d[i], x[i]);
        const float rn = fmaf(-a, q[i], r[i]);
        r[i] = rn;
        dot += (double)rn * (double)rn;
    }
    const double b = block_sum_f64(dot);
    if (threadIdx.x == 0) partial[blockIdx.x] = b;
}

// d = r + beta_cg d
__global__ void __launch_bounds__(256) map_dir_kernel(float* __restrict__ d, const float* __restrict__ r,
                                                      const double* __restrict__ scal, size_t N) {
    const float b = (float)scal[2];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x)
        d[i] = fmaf(b, d[i], r[i]);
}

enum MapFin { MFIN_RR0 = 0, MFIN_ALPHA = 1, MFIN_BETA = 2 };

// scal = {rr, alpha, beta}: one block sums the MAP_BLOCKS partials in a fixed order.
template <int MODE>
__global__ void map_finalize_kernel(const double* __restrict__ partial, double* __restrict__ scal,
                                    int* __restrict__ status) {
    double s = 0.0;
    for (int i = threadIdx.x; i < MAP_BLOCKS; i += blockDim.x) s += partial[i];
    s = block_sum_f64(s);
    if (threadIdx.x == 0) {
        if (!isfinite(s)) atomicExch(status, (int)MSF_ERR_NUMERIC);
        if (MODE == MFIN_RR0) {
            scal[0] = s;
        } else if (MODE == MFIN_ALPHA) {
            scal[1] = (s != 0.0) ? scal[0] / s : 0.0;
        } else {
            scal[2] = (scal[0] != 0.0) ? s / scal[0] : 0.0;
            scal[0] = s;
        }
    }
}

// Sinogram weighting: RES: s = Lambda (y - s); LAM: s = Lambda s; COST: partial
// sums of Lambda (y - s)^2.
enum MapSino { MS_RES = 0, MS_LAM = 1, MS_COST = 2 };
template <int MODE>
__global__ void __launch_bounds__(256) map_sino_kernel(float* __restrict__ s, const float* __restrict__ y,
                                                       const float* __restrict__ lam, size_t M,
                                                       double* __restrict__ partial) {
    double acc = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < M; i += (size_t)gridDim.x * blockDim.x) {
        if (MODE == MS_RES) {
            s[i] = lam[i] * (y[i] - s[i]);
        } else if (MODE == MS_LAM) {
            s[i] = lam[i] * s[i];
        } else {
            const double e = (double)y[i] - (double)s[i];
            acc += (double)lam[i] * e * e;
        }
    }
    if (MODE == MS_COST) {
        const double b = block_sum_f64(acc);
        if (threadIdx.x == 0) partial[blockIdx.x] = b;
    }
}

// rho(D) = D^2/(2 sx^2) * u/(1+u), u = |D/(T sx)|^(q-2)  (p = 2), in FP64.
__device__ __forceinline__ double qggmrf_rho64(double D, double q, double tsx, double sx) {
    const double ad = fabs(D);
    if (ad == 0.0) return 0.0;
    const double u = pow(ad / tsx, q - 2.0);
    return D * D / (2.0 * sx * sx) * (u / (1.0 + u));
}

// Partial sums of h(x) = sum over unordered neighbour pairs b_sr rho(x_s - x_r)
// (each pair once: the neighbours at a positive lexicographic offset).
__global__ void __launch_bounds__(256) map_prior_cost_kernel(const float* __restrict__ x, MrfDims m, double q,
                                                             double T, double sx, double* __restrict__ partial) {
    const size_t sxy = (size_t)m.nx * m.ny, fs = sxy * m.nz, N = fs * m.nt;
    const double s_ = 6.0 + 12.0 / sqrt(2.0) + 8.0 / sqrt(3.0);
    const double bf = 1.0 / s_, be = 1.0 / (sqrt(2.0) * s_), bc = 1.0 / (sqrt(3.0) * s_);
    double acc = 0.0;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < N; s += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(s / fs);
        const size_t r0 = s - (size_t)t * fs;
        const int iz = (int)(r0 / sxy);
        const int rr = (int)(r0 - (size_t)iz * sxy);
        const int iy = rr / m.nx, ix = rr - iy * m.nx;
        const double xs = x[s];
        for (int dz = 0; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
                for (int dx = -1; dx <= 1; ++dx) {
                    const bool pos = dz > 0 || (dy > 0 || (dy == 0 && dx > 0));
                    if (!pos) continue;
                    const int jx = ix + dx, jy = iy + dy, jz = iz + dz;
                    if (jx < 0 || jx >= m.nx || jy < 0 || jy >= m.ny || jz >= m.nz) continue;
                    const int mm = (dx != 0) + (dy != 0) + (dz != 0);
                    const double b = mm == 1 ? bf : (mm == 2 ? be : bc);
                    acc += b * qggmrf_rho64(xs - (double)x[(size_t)t * fs + (size_t)jz * sxy + (size_t)jy * m.nx + jx],
                                            q, T * sx, sx);
                }
        if (t + 1 < m.nt) acc += (double)m.bt * qggmrf_rho64(xs - (double)x[s + fs], q, T * sx, sx);
    }
    const double b = block_sum_f64(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = b;
}

__global__ void map_cost_finalize_kernel(const double* __restrict__ pdata, const double* __restrict__ pprior,
                                         double* __restrict__ out) {
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < MAP_BLOCKS; i += blockDim.x) {
        a += pdata[i];
        b += pprior[i];
    }
    a = block_sum_f64(a);
    b = block_sum_f64(b);
    if (threadIdx.x == 0) {
        out[0] = a;
        out[1] = b;
    }
}

static msf_status mrf_dims(const msf_vol* vol, const msf_mrf* prm, double sigma, MrfDims* out) {
    MSF_REQUIRE(prm->p == 2.0 && prm->q >= 1.0 && prm->q <= 2.0,
                "q-GGMRF: need p == 2 and 1 <= q <= 2 (got p=%g q=%g)", prm->p, prm->q);
    MSF_REQUIRE(prm->T > 0 && prm->sigma_x > 0 && prm->b_temporal >= 0,
                "q-GGMRF: T and sigma_x must be positive and b_temporal >= 0");
    MrfDims& m = *out;
    m.nx = vol->nx; m.ny = vol->ny; m.nz = vol->nz; m.nt = vol->nt;
    m.px = m.py = m.pz = m.pt = 0;
    m.hx = m.hy = m.hz = m.ht = 0;
    m.inv_s2 = (float)(1.0 / (sigma * sigma));
    m.inv_tsx = (float)(1.0 / (prm->T * prm->sigma_x));
    m.pq = (float)(prm->p - prm->q);
    const double s = 6.0 + 12.0 / sqrt(2.0) + 8.0 / sqrt(3.0), c = 1.0 / (prm->sigma_x * prm->sigma_x);
    const double b[4] = {1.0 / s, 1.0 / (sqrt(2.0) * s), 1.0 / (sqrt(3.0) * s), prm->b_temporal};
    // (a temporal weight so small that it loses bits is nothing beside the spatial ones)
    const double q1 = prm->q / prm->p;
    m.kind = prm->p - prm->q < 0.2 ? MRF_NEAR : c * (1.0 - q1) >= 0x1p-54 ? MRF_USUAL : MRF_APART;
    const double s1 = m.kind == MRF_USUAL ? MRF_SCALE : 1.0;
    for (int k = 0; k < 4; ++k) {
        m.k1[k] = (float)(b[k] * c * q1 * s1);
        m.k2[k] = (float)(b[k] * c * (1.0 - q1) * s1 * s1);
    }
    m.bt = (float)prm->b_temporal;
    return MSF_OK;
}

}  // namespace msf

struct msf_map {
    msf_projector* proj = nullptr;
    msf_vol vol;
    size_t N = 0, M = 0;
    float *d_r = nullptr, *d_d = nullptr, *d_q = nullptr, *d_anchor = nullptr, *d_s = nullptr;
    double *d_part = nullptr, *d_part2 = nullptr, *d_scal = nullptr, *d_cost = nullptr;
    double* h_cost = nullptr;   // pinned [2]
    int* d_status = nullptr;
    int* h_status = nullptr;    // pinned
};

using namespace msf;

extern "C" msf_status msf_map_create(msf_projector* p, msf_map** out) {
    MSF_REQUIRE(p && out, "msf_map_create: NULL argument");
    *out = nullptr;
    MSF_TRY(check_device());
    msf_map* m = new msf_map();
    m->proj = p;
    m->vol = *projector_volume(p);
    m->N = (size_t)m->vol.nx * m->vol.ny * m->vol.nz * m->vol.nt;
    m->M = projector_sino_size(p);
    if (cudaMalloc(&m->d_r, m->N * 4) != cudaSuccess || cudaMalloc(&m->d_d, m->N * 4) != cudaSuccess ||
        cudaMalloc(&m->d_q, m->N * 4) != cudaSuccess || cudaMalloc(&m->d_anchor, m->N * 4) != cudaSuccess ||
        cudaMalloc(&m->d_s, m->M * 4) != cudaSuccess || cudaMalloc(&m->d_part, MAP_BLOCKS * 8) != cudaSuccess ||
        cudaMalloc(&m->d_part2, MAP_BLOCKS * 8) != cudaSuccess || cudaMalloc(&m->d_scal, 4 * 8) != cudaSuccess ||
        cudaMalloc(&m->d_cost, 2 * 8) != cudaSuccess || cudaMalloc(&m->d_status, sizeof(int)) != cudaSuccess ||
        cudaMallocHost(&m->h_cost, 2 * 8) != cudaSuccess || cudaMallocHost(&m->h_status, sizeof(int)) != cudaSuccess ||
        cudaMemset(m->d_status, 0, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        msf_map_destroy(m);
        return fail(MSF_ERR_NOMEM, "msf_map_create: out of device memory");
    }
    const msf_status st = settle_default_stream();
    if (st != MSF_OK) {
        msf_map_destroy(m);
        return st;
    }
    *out = m;
    return MSF_OK;
}

extern "C" void msf_map_destroy(msf_map* m) {
    if (!m) return;
    cudaFree(m->d_r); cudaFree(m->d_d); cudaFree(m->d_q); cudaFree(m->d_anchor); cudaFree(m->d_s);
    cudaFree(m->d_part); cudaFree(m->d_part2); cudaFree(m->d_scal); cudaFree(m->d_cost); cudaFree(m->d_status);
    if (m->h_cost) cudaFreeHost(m->h_cost);
    if (m->h_status) cudaFreeHost(m->h_status);
    delete m;
}

extern "C" msf_status msf_map_solve(msf_map* m, const msf_mrf* prm, double beta, const float* d_y,
                                    const float* d_lambda, float* d_x, int n_outer, int n_cg, void* stream) {
    MSF_REQUIRE(m && prm && d_y && d_lambda && d_x, "msf_map_solve: NULL argument");
    MSF_REQUIRE(beta > 0 && isfinite(beta), "msf_map_solve: beta must be positive");
    MSF_REQUIRE(n_outer >= 0 && n_cg >= 0, "msf_map_solve: iteration counts must be >= 0");
    MrfDims md;
    MSF_TRY(mrf_dims(&m->vol, prm, 1.0, &md));
    if (n_outer == 0 || n_cg == 0) return MSF_OK;
    cudaStream_t st = as_stream(stream);
    void* sv = reinterpret_cast<void*>(st);
    const float two_beta = (float)(2.0 * beta);
    const size_t N = m->N, M = m->M;
    for (int o = 0; o < n_outer; ++o) {
        MSF_TRY_CUDA(cudaMemcpyAsync(m->d_anchor, d_x, N * 4, cudaMemcpyDeviceToDevice, st));
        // r = A^T Lambda (y - A x) - 2 beta L_a x ; d = r ; rr = r.r
        MSF_TRY(msf_project(m->proj, d_x, m->d_s, sv));
        {
            MSF_PROF("map_sino", st);
            map_sino_kernel<MS_RES><<<MAP_BLOCKS, 256, 0, st>>>(m->d_s, d_y, d_lambda, M, nullptr);
            MSF_LAUNCH_CHECK();
        }
        MSF_TRY(msf_backproject(m->proj, m->d_s, m->d_r, sv));
        {
            MSF_PROF("map_lap", st);
            launch_map_lap<MAP_INIT>(m->d_anchor, d_x, m->d_r, m->d_d, two_beta, md, m->d_part, st);
            MSF_LAUNCH_CHECK();
        }
        {
            MSF_PROF("map_finalize", st);
            map_finalize_kernel<MFIN_RR0><<<1, 1024, 0, st>>>(m->d_part, m->d_scal, m->d_status);
            MSF_LAUNCH_CHECK();
        }
        for (int k = 0; k < n_cg; ++k) {
            // q = A^T Lambda A d + 2 beta L_a d ; alpha = rr / d.q
            MSF_TRY(msf_project(m->proj, m->d_d, m->d_s, sv));
            {
                MSF_PROF("map_sino", st);
                map_sino_kernel<MS_LAM><<<MAP_BLOCKS, 256, 0, st>>>(m->d_s, nullptr, d_lambda, M, nullptr);
                MSF_LAUNCH_CHECK();
            }
            MSF_TRY(msf_backproject(m->proj, m->d_s, m->d_q, sv));
            {
                MSF_PROF("map_lap", st);
                launch_map_lap<MAP_Q>(m->d_anchor, m->d_d, m->d_q, nullptr, two_beta, md, m->d_part, st);
                MSF_LAUNCH_CHECK();
            }
            {
                MSF_PROF("map_finalize", st);
                map_finalize_kernel<MFIN_ALPHA><<<1, 1024, 0, st>>>(m->d_part, m->d_scal, m->d_status);
                MSF_LAUNCH_CHECK();
            }
            {   // x += alpha d ; r -= alpha q
                MSF_PROF("map_update", st);
                map_update_kernel<<<MAP_BLOCKS, 256, 0, st>>>(d_x, m->d_r, m->d_d, m->d_q, m->d_scal, N, m->d_part);
                MSF_LAUNCH_CHECK();
            }
            {   // beta_cg = r.r / rr
                MSF_PROF("map_finalize", st);
                map_finalize_kernel<MFIN_BETA><<<1, 1024, 0, st>>>(m->d_part, m->d_scal, m->d_status);
                MSF_LAUNCH_CHECK();
            }
            {   // d = r + beta_cg d
                MSF_PROF("map_dir", st);
                map_dir_kernel<<<MAP_BLOCKS, 256, 0, st>>>(m->d_d, m->d_r, m->d_scal, N);
                MSF_LAUNCH_CHECK();
            }
        }
    }
    return MSF_OK;
}

extern "C" msf_status msf_map_cost(msf_map* m, const msf_mrf* prm, double beta, const float* d_y,
                                   const float* d_lambda, const float* d_x, double* h_cost, void* stream) {
    MSF_REQUIRE(m && prm && d_y && d_lambda && d_x && h_cost, "msf_map_cost: NULL argument");
    MrfDims md;
    MSF_TRY(mrf_dims(&m->vol, prm, 1.0, &md));
    cudaStream_t st = as_stream(stream);
    MSF_TRY(msf_project(m->proj, d_x, m->d_s, reinterpret_cast<void*>(st)));
    {
        MSF_PROF("map_cost", st);
        map_sino_kernel<MS_COST><<<MAP_BLOCKS, 256, 0, st>>>(m->d_s, d_y, d_lambda, m->M, m->d_part);
        MSF_LAUNCH_CHECK();
    }
    {
        MSF_PROF("map_cost", st);
        map_prior_cost_kernel<<<MAP_BLOCKS, 256, 0, st>>>(d_x, md, prm->q, prm->T, prm->sigma_x, m->d_part2);
        MSF_LAUNCH_CHECK();
    }
    {
        MSF_PROF("map_cost", st);
        map_cost_finalize_kernel<<<1, 1024, 0, st>>>(m->d_part, m->d_part2, m->d_cost);
        MSF_LAUNCH_CHECK();
    }
    MSF_TRY_CUDA(cudaMemcpyAsync(m->h_cost, m->d_cost, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    MSF_TRY_CUDA(cudaMemcpyAsync(m->h_status, m->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
    MSF_TRY_CUDA(cudaStreamSynchronize(st));
    if (*m->h_status != 0) return fail(MSF_ERR_NUMERIC, "msf_map_solve: a non-finite CG scalar occurred");
    h_cost[0] = 0.5 * m->h_cost[0] + beta * m->h_cost[1];
    return MSF_OK;
}

extern "C" msf_status msf_prox_qggmrf(const msf_vol* vol, const msf_mrf* prm, const float* d_v, float* d_x,
                                      double sigma, int n_sweeps, void* stream) {
    MSF_REQUIRE(vol && prm && d_v && d_x, "msf_prox_qggmrf: NULL argument");
    MSF_REQUIRE(vol->nx > 0 && vol->ny > 0 && vol->nz > 0 && vol->nt > 0,
                "msf_prox_qggmrf: volume sizes must be positive");
    MSF_REQUIRE(prm->p == 2.0 && prm->q >= 1.0 && prm->q <= 2.0,
                "msf_prox_qggmrf: need p == 2 and 1 <= q <= 2 (got p=%g q=%g)", prm->p, prm->q);
    MSF_REQUIRE(prm->T > 0 && prm->sigma_x > 0 && prm->b_temporal >= 0 && sigma > 0,
                "msf_prox_qggmrf: T, sigma_x, sigma must be positive and b_temporal >= 0");
    MSF_REQUIRE(n_sweeps >= 0, "msf_prox_qggmrf: n_sweeps must be >= 0");
    MSF_REQUIRE((long long)((vol->nz + 1) / 2) * ((vol->nt + 1) / 2) <= 65535,
                "msf_prox_qggmrf: nz*nt too large for the launch grid");
    cudaStream_t st = as_stream(stream);
    MrfDims m;
    MSF_TRY(mrf_dims(vol, prm, sigma, &m));
    if (n_sweeps == 0) return MSF_OK;
    const long long colour = (long long)((m.nx + 1) / 2) * ((m.ny + 1) / 2) * ((m.nz + 1) / 2) * ((m.nt + 1) / 2);
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) cudaGetLastError();   // (a launch will report it)
    if (colour <= ICD_SMALL_VOXELS && capture == cudaStreamCaptureStatusNone) {
        MSF_PROF("qggmrf_icd", st);
        auto* f = m.kind == MRF_USUAL ? icd_small_kernel<MRF_USUAL>
                  : m.kind == MRF_NEAR ? icd_small_kernel<MRF_NEAR> : icd_small_kernel<MRF_APART>;
        f<<<ICD_CLUSTER, ICD_SMALL_THREADS, 0, st>>>(d_v, d_x, m, n_sweeps);
        MSF_LAUNCH_CHECK();
        return MSF_OK;
    }
    for (int sw = 0; sw < n_sweeps; ++sw) {
        for (int col = 0; col < 16; ++col) {
            m.px = col & 1; m.py = (col >> 1) & 1; m.pz = (col >> 2) & 1; m.pt = (col >> 3) & 1;
            m.hx = (m.nx - m.px + 1) / 2; m.hy = (m.ny - m.py + 1) / 2;
            m.hz = (m.nz - m.pz + 1) / 2; m.ht = (m.nt - m.pt + 1) / 2;
            if (m.hx <= 0 || m.hy <= 0 || m.hz <= 0 || m.ht <= 0) continue;
            dim3 grid((m.hx + 31) / 32, (m.hy + 3) / 4, m.hz * m.ht);
            MSF_PROF("qggmrf_icd", st);
            // the twelve blocks of every SM
            const bool deep = (long long)grid.x * grid.y * grid.z >= 12 * 152;
            auto* f = m.kind == MRF_APART  ? icd_colour_kernel<MRF_APART, 1>
                      : m.kind == MRF_NEAR ? (deep ? icd_colour_kernel<MRF_NEAR, 12> : icd_colour_kernel<MRF_NEAR, 1>)
                                           : (deep ? icd_colour_kernel<MRF_USUAL, 12> : icd_colour_kernel<MRF_USUAL, 1>);
            f<<<grid, dim3(32, 4), 0, st>>>(d_v, d_x, m);
            MSF_LAUNCH_CHECK();
        }
    }
    return MSF_OK;
}
