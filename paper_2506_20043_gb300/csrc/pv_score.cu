// pv_score.cu -- batched scoring of given poses (Eq. 3) with the adjoint gradient, one warp per
// pose; the vector-Jacobian product used by automatic differentiation; forward kinematics only.
#include <algorithm>

#include "pv_internal.h"
#include "pv_smem.h"
#include "pv_stage.cuh"
#include "pv_warp.cuh"

namespace pv {

// One CTA per SM, of up to 28 warps (72 registers each), a warp per pose: the ligand is staged once per SM, and
// the number of warps is chosen so that every warp takes the same number of poses (score_shape below). CTAs of
// 8 warps, three per SM (73 registers), staged it three times and left a last wave of a few poses per SM, and a
// launch asked for its occupancy: 65,536 poses of a 32-atom ligand 120.5 -> 108 us a pass; 8,191 poses
// of 47 atoms 43 -> 39 us, 64 poses of 20 atoms 7.7 -> 6.2 us of device time.
constexpr int kScoreWarps = 28;
constexpr int kScoreLeastWarps = 4;    // below that staging the ligand takes longer than the poses

struct ScoreArgs {
    const PvLigBlob* lig;
    int lig_bytes;
    const PvPocket* pocket;
    uint64_t slots_lo, slots_hi;
    int n_poses, pot_stride;
    const float* pose;
    float* energy;        // forward outputs (nullable)
    float* grad;
    float* parts;
    const float* grad_energy;   // backward: scale of the two below (null: 1)
    float* grad_pose;           // nullable
    float* grad_xyz;
    int fk_only;
    float* xyz;
};

__device__ __forceinline__ Pose read_pose(const float* p, int n_rot) {
    const int lane = threadIdx.x & 31;
    Pose x;
    x.T = make_float3(p[0], p[1], p[2]);
    x.q = make_float4(p[3], p[4], p[5], p[6]);
    x.psi = (lane >= 6 && lane < 6 + n_rot) ? p[lane + 1] : 0.f;
    return x;
}

template <int LAYOUT>
__global__ void __launch_bounds__(kScoreWarps * 32, 1) score_kernel(ScoreArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    PvLigBlob& L = *reinterpret_cast<PvLigBlob*>(smem);
    WarpScratch* scratch = reinterpret_cast<WarpScratch*>(smem + ((A.lig_bytes + 127) & ~127));
    __shared__ PvPocket s_pocket;
    if (!A.fk_only && threadIdx.x < (int)(sizeof(PvPocket) / 4))
        reinterpret_cast<int*>(&s_pocket)[threadIdx.x] = reinterpret_cast<const int*>(A.pocket)[threadIdx.x];
    stage_ligand(&L, A.lig, A.slots_lo, A.slots_hi);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int n_rot = L.h.n_rot, n = L.h.n_atoms, nt = 6 + n_rot;
    WarpScratch& S = scratch[warp];
    init_scratch<32>(S);
    Site site;
    site.maps = s_pocket.maps;
    site.P = &s_pocket;
    for (int i = blockIdx.x * W + warp; i < A.n_poses; i += gridDim.x * W) {
        const float* p = A.pose + (size_t)i * A.pot_stride;
        const Pose x = read_pose(p, n_rot);
        if (A.fk_only) {
            float3 axw, xa;
            warp_fk(L, S, x, axw, xa);
            __syncwarp();
            for (int a = lane; a < n; a += 32) {
                float* dst = A.xyz + ((size_t)i * n + L.atom_src[a]) * 3;
                dst[0] = S.x[a].x; dst[1] = S.x[a].y; dst[2] = S.x[a].z;
            }
            __syncwarp();
            continue;
        }
        const bool want_grad = A.grad || A.grad_pose || A.grad_xyz;
        float g = 0.f, parts[2];
        const float e = warp_eval<LAYOUT>(L, S, site, x, g, want_grad, parts);
        if (A.energy && lane == 0) A.energy[i] = e;
        if (A.parts && lane == 0) { A.parts[2 * i] = parts[0]; A.parts[2 * i + 1] = parts[1]; }
        if (A.grad && lane < nt) A.grad[(size_t)i * nt + lane] = g;
        if (A.grad_pose || A.grad_xyz) {
            const float dE = A.grad_energy ? A.grad_energy[i] : 1.f;
            if (A.grad_pose) {
                float* out = A.grad_pose + (size_t)i * A.pot_stride;
                // translation
                if (lane < 3) out[lane] = dE * g;
                // raw quaternion through the normalisation: with unit (w, v) = q / |q| and the
                // world rotation gradient G, dSF/dq_w = -2 v.G / |q|, dSF/dv = 2 (w G + G x v) / |q|
                const float3 G = make_float3(shfl(g, 3), shfl(g, 4), shfl(g, 5));
                const float qn = sqrtf(x.q.x * x.q.x + x.q.y * x.q.y + x.q.z * x.q.z + x.q.w * x.q.w);
                const float w = x.q.x / qn;
                const float3 v = make_float3(x.q.y / qn, x.q.z / qn, x.q.w / qn);
                const float3 gv = (2.f / qn) * (w * G + cross3(G, v));
                const float gw = -2.f / qn * dot3(v, G);
                if (lane == 3) out[3] = dE * gw;
                if (lane == 4) out[4] = dE * gv.x;
                if (lane == 5) out[5] = dE * gv.y;
                if (lane == 6) out[6] = dE * gv.z;
                if (lane >= 6 && lane < nt) out[lane + 1] = dE * g;
            }
            if (A.grad_xyz) {
                for (int a = lane; a < n; a += 32) {
                    float* dst = A.grad_xyz + ((size_t)i * n + L.atom_src[a]) * 3;
                    const float4 gg = S.g[a];
                    dst[0] = dE * gg.x; dst[1] = dE * gg.y; dst[2] = dE * gg.z;
                }
            }
        }
        __syncwarp();
    }
}

// CTA size and grid for n poses: as few rounds of the resident warps as they need, then as few warps as do them
// in that many rounds.
struct ScoreShape {
    int warps, grid, smem;
};
static cudaError_t score_shape(int dev, int n, int lig_bytes, ScoreShape& s) {
    static DevicePair properties;
    int n_sm = 0, smem_max = 0;
    const int e = properties.get(dev, n_sm, smem_max, [dev](int& sms, int& smem) {
        const cudaError_t x = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        return (int)(x != cudaSuccess ? x : cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    });
    if (e) return (cudaError_t)e;
    const int lig = (lig_bytes + 127) & ~127;
    const int most = std::min(kScoreWarps, (smem_max - 1024 - lig) / (int)sizeof(WarpScratch));
    if (most < 1) return cudaErrorInvalidValue;
    const int rounds = (n + n_sm * most - 1) / (n_sm * most);
    s.warps = std::max(std::min(most, kScoreLeastWarps), (n + n_sm * rounds - 1) / (n_sm * rounds));
    s.grid = std::min(n_sm, (n + s.warps - 1) / s.warps);
    s.smem = lig + s.warps * (int)sizeof(WarpScratch);
    return cudaSuccess;
}

// The shape of a launch on the current device, and the kernel's shared-memory limit raised to it.
static cudaError_t score_setup(const void* fn, SmemLimit& limit, int n, int lig_bytes, ScoreShape& s) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidValue;
    e = score_shape(dev, n, lig_bytes, s);
    if (e != cudaSuccess) return e;
    return (cudaError_t)limit.raise(dev, s.smem, [fn](int bytes) {
        return (int)cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    });
}

static cudaError_t launch(const ScoreArgs& a, int layout, cudaStream_t s) {
    if (layout < 0 || layout > 1) return cudaErrorInvalidValue;
    if (a.n_poses < 1) return cudaSuccess;
    static SmemLimit limit[2];
    const void* fn = layout == 1 ? (const void*)score_kernel<1> : (const void*)score_kernel<0>;
    ScoreShape sh;
    const cudaError_t e = score_setup(fn, limit[layout], a.n_poses, a.lig_bytes, sh);
    if (e != cudaSuccess) return e;
    if (layout == 1) score_kernel<1><<<sh.grid, sh.warps * 32, sh.smem, s>>>(a);
    else score_kernel<0><<<sh.grid, sh.warps * 32, sh.smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_score(const PvLigBlob* lig, int lig_bytes, const PvPocket* pocket,
                         PvSlots slots, int n_poses, int pot_stride,
                         const float* pose, float* energy, float* grad, float* parts,
                         const float* grad_energy, float* grad_pose, float* grad_xyz,
                         int layout, cudaStream_t s) {
    ScoreArgs a{};
    a.lig = lig; a.lig_bytes = lig_bytes; a.pocket = pocket;
    uint64_t lo = 0, hi = 0;
    for (int t = 0; t < 16; ++t) {
        uint64_t b = (uint64_t)(uint8_t)slots.slot[t];
        if (t < 8) lo |= b << (8 * t); else hi |= b << (8 * (t - 8));
    }
    a.slots_lo = lo; a.slots_hi = hi;
    a.n_poses = n_poses; a.pot_stride = pot_stride; a.pose = pose;
    a.energy = energy; a.grad = grad; a.parts = parts;
    a.grad_energy = grad_energy; a.grad_pose = grad_pose; a.grad_xyz = grad_xyz;
    return launch(a, layout, s);
}

// SF of posed ligands given by their atom coordinates (input order), one warp per ligand: the atoms
// go to S.x in device order, then the same interpolation and pair rounds as for a pose; the
// coordinate gradient, scaled by grad_energy when given, comes from S.g.
struct ScoreXyzArgs {
    const PvLigBlob* lig;
    int lig_bytes;
    const PvPocket* pocket;
    uint64_t slots_lo, slots_hi;
    int n_poses;
    const float* xyz;
    const float* grad_energy;   // nullable: scale 1
    float* energy;              // nullable
    float* grad_xyz;            // nullable
};

template <int LAYOUT>
__global__ void __launch_bounds__(kScoreWarps * 32, 1) score_xyz_kernel(ScoreXyzArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    PvLigBlob& L = *reinterpret_cast<PvLigBlob*>(smem);
    WarpScratch* scratch = reinterpret_cast<WarpScratch*>(smem + ((A.lig_bytes + 127) & ~127));
    __shared__ PvPocket s_pocket;
    if (threadIdx.x < (int)(sizeof(PvPocket) / 4))
        reinterpret_cast<int*>(&s_pocket)[threadIdx.x] = reinterpret_cast<const int*>(A.pocket)[threadIdx.x];
    stage_ligand(&L, A.lig, A.slots_lo, A.slots_hi);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int n = L.h.n_atoms;
    WarpScratch& S = scratch[warp];
    init_scratch<32>(S);
    Site site;
    site.maps = s_pocket.maps;
    site.P = &s_pocket;
    const Pose none{};
    for (int i = blockIdx.x * W + warp; i < A.n_poses; i += gridDim.x * W) {
        for (int a = lane; a < n; a += 32) {
            const float* src = A.xyz + ((size_t)i * n + L.atom_src[a]) * 3;
            const int t = (__float_as_int(L.atom[a].w) >> 8) & 255;
            S.x[a] = make_float4(src[0], src[1], src[2], xs_radius(t));
        }
        __syncwarp();
        float g = 0.f;
        const float e = team_eval<32, false, LAYOUT>(L, S, site, none, g, false);
        if (A.energy && lane == 0) A.energy[i] = e;
        if (A.grad_xyz) {
            const float s = A.grad_energy ? A.grad_energy[i] : 1.f;
            for (int a = lane; a < n; a += 32) {
                float* dst = A.grad_xyz + ((size_t)i * n + L.atom_src[a]) * 3;
                const float4 gg = S.g[a];
                dst[0] = s * gg.x; dst[1] = s * gg.y; dst[2] = s * gg.z;
            }
        }
        __syncwarp();
    }
}

cudaError_t launch_score_xyz(const PvLigBlob* lig, int lig_bytes, const PvPocket* pocket, PvSlots slots,
                             int n_poses, const float* xyz, const float* grad_energy, float* energy,
                             float* grad_xyz, int layout, cudaStream_t s) {
    ScoreXyzArgs a{};
    a.lig = lig; a.lig_bytes = lig_bytes; a.pocket = pocket;
    uint64_t lo = 0, hi = 0;
    for (int t = 0; t < 16; ++t) {
        uint64_t b = (uint64_t)(uint8_t)slots.slot[t];
        if (t < 8) lo |= b << (8 * t); else hi |= b << (8 * (t - 8));
    }
    a.slots_lo = lo; a.slots_hi = hi;
    a.n_poses = n_poses; a.xyz = xyz; a.grad_energy = grad_energy; a.energy = energy; a.grad_xyz = grad_xyz;
    if (layout < 0 || layout > 1) return cudaErrorInvalidValue;
    if (n_poses < 1) return cudaSuccess;
    static SmemLimit limit[2];
    const void* fn = layout == 1 ? (const void*)score_xyz_kernel<1> : (const void*)score_xyz_kernel<0>;
    ScoreShape sh;
    const cudaError_t e = score_setup(fn, limit[layout], n_poses, lig_bytes, sh);
    if (e != cudaSuccess) return e;
    if (layout == 1) score_xyz_kernel<1><<<sh.grid, sh.warps * 32, sh.smem, s>>>(a);
    else score_xyz_kernel<0><<<sh.grid, sh.warps * 32, sh.smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_pose_coords(const PvLigBlob* lig, int lig_bytes, int n_poses, int pot_stride,
                               const float* pose, float* xyz, cudaStream_t s) {
    ScoreArgs a{};
    a.lig = lig; a.lig_bytes = lig_bytes; a.n_poses = n_poses; a.pot_stride = pot_stride;
    a.pose = pose; a.fk_only = 1; a.xyz = xyz;
    return launch(a, 0, s);
}

}  // namespace pv
