// Shared by the projector's two layouts (projector.cu: volumes in lines along z;
// projector_planes.cu: volumes in planes of z-pairs): ray constants, the data agents'
// scalars, and the plan and workspace handles.
#pragma once

#include <vector>

#include "common.cuh"

namespace msf {

struct ColParams {
    float fa_mid, ba, c1, inv_dmaj;   // minor-axis line, z factors
    float dxy2, vox_over_adm, xmajor, pad;
};

struct ProjDims {
    int nx, ny, nz, nt, nu, nv, views;
    float cx, cy, cz, cu, cv;   // (n-1)/2 of each axis
    float vox, du, dv;
    float dso, dsd;
};

struct RayZ {
    float fz_mid, bz, step;
};

// The one place where a ray's z constants are formed; forward and adjoint
// both call it, with explicit round-to-nearest intrinsics so the compiler
// cannot contract the two call sites differently.
__device__ __forceinline__ RayZ ray_z(const ColParams& c, float v, float cz) {
    RayZ r;
    r.fz_mid = __fmaf_rn(v, c.c1, cz);
    r.bz = __fmul_rn(v, c.inv_dmaj);
    r.step = __fmul_rn(__fsqrt_rn(__fmaf_rn(v, v, c.dxy2)), c.vox_over_adm);
    return r;
}

__device__ __forceinline__ float det_v(int iv, const ProjDims& d) {
    return __fmul_rn(__fsub_rn((float)iv, d.cv), d.dv);
}

__device__ __forceinline__ ColParams load_col(const float4* __restrict__ col, size_t idx) {
    float4 a = __ldg(col + 2 * idx), b = __ldg(col + 2 * idx + 1);
    ColParams c;
    c.fa_mid = a.x; c.ba = a.y; c.c1 = a.z; c.inv_dmaj = a.w;
    c.dxy2 = b.x; c.vox_over_adm = b.y; c.xmajor = b.z; c.pad = b.w;
    return c;
}

// Detector u coordinate (in pixels) of the point (x, y, .) for view (cs, sn);
// only used to bound candidate columns, so a fast division is enough.
__device__ __forceinline__ float u_pixel(float x, float y, float cs, float sn, const ProjDims& d) {
    const float lat = -x * sn + y * cs;
    const float depth = d.dso - x * cs - y * sn;
    return __fdividef(d.dsd * lat, depth * d.du) + d.cu;
}

enum FwdMode { FWD_PLAIN = 0, FWD_LAMBDA = 1, FWD_RESIDUAL = 2, FWD_ICD = 3 };

enum AdjMode { ADJ_PLAIN = 0, ADJ_CG_INIT = 1, ADJ_CG_Q = 2, ADJ_THETA2 = 3 };

// ------------------------------------------------------------------ CG scalars
//
// A kernel whose blocks each hold a partial sum of a frame hands them to the
// frame's last block, which adds them in a fixed order and forms the scalar:
//   FIN_RR0:   rr = sum
//   FIN_ALPHA: alpha = rr / sum (0 when sum == 0)
//   FIN_BETA:  beta = sum / rr (0 when rr == 0); rr = sum
// Any non-finite sum raises the status flag.  (A kernel of its own per scalar
// cost a launch, 11 per five CG steps.)
enum FinMode { FIN_RR0 = 0, FIN_ALPHA = 1, FIN_BETA = 2 };

struct CgScalars {
    double* partial;      // [nt][blocks of a frame]
    double *rr, *coef;    // [nt]
    int* status;
    unsigned* count;      // [nt], zero between kernels: blocks of the frame that have stored their sum
};

// sum: this block's partial, in thread 0; b of nparts: its place in frame t.
template <int FIN>
__device__ __forceinline__ void frame_finalize(double sum, int t, int b, int nparts, const CgScalars& c) {
    __shared__ bool last;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y, nthreads = blockDim.x * blockDim.y;
    double* part = c.partial + (size_t)t * nparts;
    if (tid == 0) {
        part[b] = sum;
        __threadfence();
        last = atomicAdd(c.count + t, 1u) == (unsigned)nparts - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (int i = tid; i < nparts; i += nthreads) s += __ldcg(part + i);
    s = block_sum_f64(s);
    if (tid == 0) {
        if (!isfinite(s)) atomicExch(c.status, (int)MSF_ERR_NUMERIC);
        if (FIN == FIN_RR0) {
            c.rr[t] = s;
        } else if (FIN == FIN_ALPHA) {
            c.coef[t] = (s != 0.0) ? c.rr[t] / s : 0.0;
        } else {
            c.coef[t] = (c.rr[t] != 0.0) ? s / c.rr[t] : 0.0;
            c.rr[t] = s;
        }
        c.count[t] = 0;
    }
}

// Group dimensions: voxels of parity p along an axis of n voxels.
__host__ __device__ __forceinline__ int par_count(int n, int p) { return (n - p + 1) / 2; }

struct IcdGroup {
    int px, py, pz;
    int gx, gy, gz;   // group voxels along x, y, z
};

// Sums of a group step: per frame, theta1.delta and delta.delta of the gather's
// blocks, Lambda (A delta)^2 of the forward's, and the line search's scalar
//   alpha_t = -sum(theta1.delta) / (sum Lambda (A delta)^2 + sum(delta.delta)/sigma^2).
struct IcdSums {
    double *gpart, *spart;   // [nt][gblocks][2], [nt][blocks of a frame's forward]
    int gblocks;
    double* alpha;           // [nt]
    double inv_s2;
    int* status;
    unsigned* count;         // [nt], zero between kernels
};

// The sum of a forward block's Lambda (A delta)^2 (in thread 0); the frame's last
// block forms alpha_t from the partials of both kernels in a fixed order.
__device__ __forceinline__ void icd_alpha(double sum, int t, int b, int nparts, const IcdSums& S) {
    __shared__ bool last;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y, nthreads = blockDim.x * blockDim.y;
    double* part = S.spart + (size_t)t * nparts;
    if (tid == 0) {
        part[b] = sum;
        __threadfence();
        last = atomicAdd(S.count + t, 1u) == (unsigned)nparts - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double gd = 0.0, dd = 0.0, sq = 0.0;
    for (int i = tid; i < S.gblocks; i += nthreads) {
        gd += S.gpart[2 * ((size_t)t * S.gblocks + i)];
        dd += S.gpart[2 * ((size_t)t * S.gblocks + i) + 1];
    }
    for (int i = tid; i < nparts; i += nthreads) sq += __ldcg(part + i);
    gd = block_sum_f64(gd);
    dd = block_sum_f64(dd);
    sq = block_sum_f64(sq);
    if (tid == 0) {
        const double den = sq + dd * S.inv_s2;
        if (!isfinite(gd) || !isfinite(den)) atomicExch(S.status, (int)MSF_ERR_NUMERIC);
        S.alpha[t] = (den > 0.0 && isfinite(den) && isfinite(gd)) ? -gd / den : 0.0;
        S.count[t] = 0;
    }
}

}  // namespace msf

struct msf_projector {
    msf_geom geom;
    msf_vol vol;
    msf::ProjDims dims;
    std::vector<double> angles;
    double* d_angles = nullptr;
    float4* d_col = nullptr;
    float2* d_trig = nullptr;
    int* d_vflag = nullptr;
    // which layout each call takes (choose_routes): lines along z, or planes of z-pairs
    // (A^T and CG together)
    bool fwd_planes = false, adj_planes = false, icd_planes = false;
    void* d_in = nullptr;      // the forward's input: d_vz, or d_px and d_py (a plan that has both keeps them in one place)
    float* d_vz = nullptr;     // lines: a volume's lines along z
    float* d_zero = nullptr;   // lines: one line of zeros
    float2* d_px = nullptr;    // planes: z-paired volume, [nt][nz][nx][ny] (x-major rays)
    float2* d_py = nullptr;    // planes: z-paired volume, [nt][nz][ny][nx] (y-major rays)
    float* d_sw = nullptr;     // step-weighted sinogram for msf_backproject
    // launch shapes: columns x rows of the planes' forward blocks (lines: fwd_cols, detector
    // columns per block) and z-run of the planes' gather (lines: adj_j, voxels per lane)
    int fwd_bx = 32, fwd_by = 4;
    int adj_zb = 64;
    uint64_t tuning_gen = 0;       // advanced whenever the launch shapes change
    size_t bytes = 0;
};

struct msf_dataprox {
    msf_projector* p = nullptr;
    // Lines.  CG: residual, direction and A^T Lambda A p + p / sigma^2, as lines (d_q
    // first holds v - z; z itself runs in the plan's d_vz)
    float *d_r = nullptr, *d_p = nullptr, *d_q = nullptr;
    // step-weighted sinograms in lines of rows: e' ; ICD: step Lambda (A delta) (first
    // step^2 Lambda).
    float *d_rows = nullptr, *d_rows2 = nullptr;
    // Planes.  The same vectors and sinograms in their natural order, d_p2 a second buffer of
    // the direction; the vectors are one allocation (d_r).
    float* d_p2 = nullptr;
    // ICD in lines: v, theta2 and delta, in place of CG vectors (and, of a plan whose CG
    // takes planes, in its forward's input after z)
    float *i_v = nullptr, *i_theta2 = nullptr, *i_delta = nullptr;
    double *d_partial = nullptr, *d_rr = nullptr, *d_alpha = nullptr, *d_beta = nullptr;
    int* d_status = nullptr;
    unsigned* d_count = nullptr;
    int parts_upd = 0;
    double *d_ipart = nullptr, *d_spart = nullptr;   // ICD: partial sums of the group gather and its forward
};

namespace msf {

inline size_t frame_size(const msf_vol& v) { return (size_t)v.nx * v.ny * v.nz; }
inline size_t vol_size(const msf_vol& v) { return frame_size(v) * v.nt; }
inline size_t sino_size(const msf_projector* p) {
    return (size_t)p->geom.nu * p->geom.nv * p->geom.views * p->vol.nt;
}

// ------------------------------------------------------------------ the planes' layout (projector_planes.cu)

// Whether a problem's launches stay within the grid limits there.
bool planes_fit(const ProjDims& d);
msf_status planes_project(msf_projector* p, const float* x, float* y, cudaStream_t st);
msf_status planes_backproject(msf_projector* p, const float* y, float* x, cudaStream_t st);
// The kernels of the two alone, for the autotuner: from the plan's pairs, from a
// step-weighted sinogram; and the gather's blocks per frame with z-runs of zb.
msf_status planes_project_pairs(msf_projector* p, float* y, cudaStream_t st);
msf_status planes_gather(msf_projector* p, const float* e, float* x, cudaStream_t st);
int planes_adj_blocks(const ProjDims& d, int zb);
// Workspace of the data agents (MSF_ERR_NOMEM: the caller releases it), its sinograms and
// ICD partial sums at least as large as stated; and the agents.
msf_status planes_dataprox_alloc(msf_dataprox* d, size_t sino, size_t ipart, size_t spart);
msf_status planes_prox_cg(msf_dataprox* dp, const float* y, const float* lambda, const float* v, float* x, float inv_s2,
                          int n_cg, cudaStream_t st);
msf_status planes_prox_icd(msf_dataprox* dp, const float* y, const float* lambda, const float* v, float* x, double sigma,
                           int n_sweeps, cudaStream_t st);

}  // namespace msf
