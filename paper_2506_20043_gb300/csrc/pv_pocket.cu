// pv_pocket.cu -- the pocket side of PocketVina (Methods "Pocket Prediction with P2Rank",
// Eq. 1-2, Supplementary Algorithm 1): solvent-accessible surface points of a receptor, the
// distance-weighted property sums of Eq. 1 with the protrusion count at points, and the
// single-linkage clusters of high-scoring points with their Eq. 2 scores, centres and ranking.
//
// Layout. Receptor atoms are binned into cubic cells of kCell A over their bounding box (CSR,
// input order kept within a cell, so every sum below runs in a fixed order). The SAS kernel runs
// one warp per atom: the warp gathers the atoms whose expanded spheres can reach its sphere into
// a shared-memory list, near ones first; each lane tests the lattice points lane + 32 m against the
// near ones, keeping one burial bit per point in a register, and the warp takes the few points left
// one by one against the rest. The feature kernel runs one CTA per 32 points: the atoms of the cells
// within reach of the group's bounding box are staged 32 at a time in shared memory with one chunk of
// their property columns, and every lane accumulates its point's sums in registers. Clustering hashes
// points into link-sized cells, joins neighbours with a lock-free union-find that always hooks the
// larger root under the smaller (so a component's root is its lowest index), and reduces per root in
// float64.
//
// Every step but the features runs once for all receptors or point sets of a call: blockIdx.y picks the
// item's record (SurfaceItem, ClusterItem) from a table uploaded with the inputs, so a call costs a dozen
// launches whatever the number of receptors.
//
// Device memory comes from a library-owned stream-ordered pool per device (allocated and freed on
// the context's stream); freed blocks stay in the pool for the next call.
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "pocketvina.h"
#include "pv_internal.h"
#include "pv_runs.h"

namespace {

using pv::launch_runs;
using pv::RunExtent;

constexpr int kSurfaceMagic = 0x53524631;
constexpr int kClustersMagic = 0x434c5331;
constexpr float kCell = 4.0f;            // atom binning cell edge, A
constexpr int kMaxAtoms = 200000;
constexpr int kNb = 128;                 // neighbour list capacity per warp (SAS kernel)
constexpr int kSasWarps = 4;
constexpr int kFeatSplit = 12;           // warps sharing one group of 32 points (feature kernel)
constexpr int kFeatRows = 256;           // cell rows listed at a time by the feature kernel
constexpr int kPropChunk = 8;            // property columns per feature launch row (a multiple of 4)
constexpr double kPi = 3.14159265358979323846;
constexpr int kHookRounds = 3;           // hooking rounds before the unions (clustering)

// Bondi (J. Phys. Chem. 68, 441, 1964) van der Waals radii by element: C, N, O, S.
__constant__ float c_bondi[4] = {1.70f, 1.55f, 1.52f, 1.80f};

struct AtomGrid {
    float lo[3];
    float inv_cell;
    int cd[3];
};

enum : int { kErrElement = 1, kErrRadius = 2, kErrCoord = 4, kErrUnion = 8 };

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ int cell_coord(float x, float lo, float inv, int cd) {
    return clampi(__float2int_rd((x - lo) * inv), 0, cd - 1);
}

// One lattice point of atom A (radius a): the same expression wherever a point is formed.
__device__ __forceinline__ float3 sphere_point(const float4& A, float a, const float* dirs, int k) {
    return make_float3(fmaf(a, __ldg(dirs + 3 * k), A.x), fmaf(a, __ldg(dirs + 3 * k + 1), A.y),
                       fmaf(a, __ldg(dirs + 3 * k + 2), A.z));
}

// ------------------------------------------------------------------------------ binning ---

// One receptor of a surface call (device pointers).
struct SurfaceItem {
    const float* xyz;        // [n][3]
    const uint8_t* element;
    const float* radius;     // or null: Bondi radii by element
    int n, n_cells;
    AtomGrid G;
    float reach_max;         // largest a_j plus a margin
    float4* atoms;           // input order: (x, y, z, index bits)
    float* arad;             // a_i = R_i + probe, input order
    int* key;                // cell of an atom
    int* count;              // [n_cells] atoms of a cell
    int* head;               // [n_cells] 1 + the last atom linked into the cell's list, 0: none
    int* next;               // [n] likewise
    int* cell_start;         // [n_cells + 1]
    float4* sorted;          // cell order, input order within a cell
    float* srad;             // a_i, cell order
    int* order;              // input index of the sorted atoms
    uint32_t* kept;          // [n][32]: bit m of lane's word = point lane + 32 m kept
    int* n_kept;             // [n]
    int* offset;             // [n + 1] first kept point of an atom, atoms in input order
    int* offset_sorted;      // [n + 1] the same with atoms in cell order
    float* pts;              // [n_points][3]
    int* src;                // [n_points]
    int* perm;               // [n_points] points grouped by the cell order of their atoms
    int* status;             // [0] error bits, [1] kept points
};

// Bounding box and validity of device-resident receptors, one CTA each: out[8 j ..] = lo, hi (x, y, z),
// the largest radius, error bits (kErrCoord: a coordinate beyond 1e6 A or not finite; kErrRadius).
struct BoundsItem {
    const float* xyz;
    const float* radius;
    int n;
};
__global__ void __launch_bounds__(1024) bounds_kernel(const BoundsItem* __restrict__ items, float* __restrict__ out) {
    __shared__ float s_v[8][32];
    const BoundsItem it = items[blockIdx.x];
    float v[8];
#pragma unroll
    for (int k = 0; k < 3; ++k) { v[k] = INFINITY; v[3 + k] = -INFINITY; }
    v[6] = 0.f;
    int err = 0;
    for (int i = threadIdx.x; i < it.n; i += 1024) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float x = it.xyz[3 * (size_t)i + k];
            if (!(fabsf(x) <= 1e6f)) err |= kErrCoord;
            v[k] = fminf(v[k], x);
            v[3 + k] = fmaxf(v[3 + k], x);
        }
        if (it.radius) {
            const float r = it.radius[i];
            if (!(r > 0.f && r <= 10.f)) err |= kErrRadius;
            v[6] = fmaxf(v[6], r);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    err = __reduce_or_sync(0xffffffffu, err);
    auto fold = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                const float u = __shfl_xor_sync(0xffffffffu, v[k], o);
                v[k] = k < 3 ? fminf(v[k], u) : fmaxf(v[k], u);
            }
    };
    fold();
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 7; ++k) s_v[k][warp] = v[k];
        s_v[7][warp] = __int_as_float(err);
    }
    __syncthreads();
    if (warp != 0) return;
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = s_v[k][lane];
    err = __reduce_or_sync(0xffffffffu, __float_as_int(s_v[7][lane]));
    fold();
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 7; ++k) out[8 * blockIdx.x + k] = v[k];
        out[8 * blockIdx.x + 7] = __int_as_float(err);
    }
}

// Atoms in input order, expanded radii, and each atom linked into its cell's list.
__global__ void __launch_bounds__(256) prep_atoms_kernel(const SurfaceItem* __restrict__ items, float probe) {
    const SurfaceItem& g = items[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    const float x = g.xyz[3 * i], y = g.xyz[3 * i + 1], z = g.xyz[3 * i + 2];
    float r;
    if (g.radius) {
        r = g.radius[i];
        if (!(r > 0.f && r <= 10.f)) atomicOr(g.status, kErrRadius);
    } else {
        const int e = g.element[i];
        if (e > 3) atomicOr(g.status, kErrElement);
        r = c_bondi[e & 3];
    }
    if (!(isfinite(x) && isfinite(y) && isfinite(z))) atomicOr(g.status, kErrCoord);
    g.atoms[i] = make_float4(x, y, z, __int_as_float(i));
    g.arad[i] = r + probe;
    const int c = (cell_coord(z, g.G.lo[2], g.G.inv_cell, g.G.cd[2]) * g.G.cd[1] +
                   cell_coord(y, g.G.lo[1], g.G.inv_cell, g.G.cd[1])) * g.G.cd[0] +
                  cell_coord(x, g.G.lo[0], g.G.inv_cell, g.G.cd[0]);
    g.key[i] = c;
    atomicAdd(&g.count[c], 1);
    g.next[i] = atomicExch(&g.head[c], i + 1);
}

// Exclusive scan of count(0 .. n) into start[0 .. n] by one CTA of 1024 threads, over tiles of
// 4096 elements (four consecutive elements per thread), carrying the running total, which is returned.
template <typename F>
__device__ __forceinline__ int block_scan(F&& count, int n, int* __restrict__ start) {
    __shared__ int s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int carry = 0;
    for (int base = 0; base < n; base += 4096) {
        const int i0 = base + 4 * (int)threadIdx.x;
        int v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = i0 + k < n ? count(i0 + k) : 0;
        const int sum = v[0] + v[1] + v[2] + v[3];
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();                                 // the previous tile is done with s_warp
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int w = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            s_warp[lane] = w;
        }
        __syncthreads();
        int run = carry + x - sum + (warp ? s_warp[warp - 1] : 0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i0 + k < n) start[i0 + k] = run;
            run += v[k];
        }
        carry += s_warp[31];
    }
    if (threadIdx.x == 0) start[n] = carry;
    return carry;
}

__global__ void __launch_bounds__(1024) cell_scan_kernel(const SurfaceItem* __restrict__ items) {
    const SurfaceItem& g = items[blockIdx.y];
    const int* count = g.count;
    block_scan([&](int i) { return count[i]; }, g.n_cells, g.cell_start);
}

// Every atom to its place: its cell's first slot plus the number of the cell's atoms of lower index.
__global__ void __launch_bounds__(256) sort_atoms_kernel(const SurfaceItem* __restrict__ items) {
    const SurfaceItem& g = items[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    const int c = g.key[i];
    int r = g.cell_start[c];
    for (int a = g.head[c]; a; a = g.next[a - 1]) r += a - 1 < i;
    g.sorted[r] = g.atoms[i];
    g.srad[r] = g.arad[i];
    g.order[r] = i;
}

// ---------------------------------------------------------------------- Step 1: SAS ---

// The points of atom A not yet buried, against the spheres of the list: the n_near near ones at its
// front (each buries about a third of the sphere) lane by lane, every lane its points lane + 32 m; then
// the points left (about one in ten) four at a time, eight lanes each, against the n_far others at the
// list's end. Whether a point is buried does not depend on the order of the tests.
__device__ __forceinline__ uint32_t bury(const float4* nb, int n_near, int n_far, const float4& A, float a,
                                         const float* dirs, int n_sphere, int lane, uint32_t buried) {
    const int M = (n_sphere + 31) >> 5;
    auto inside = [](const float3& p, const float4& q) {
        const float dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
        return dx * dx + dy * dy + dz * dz < q.w;
    };
    const int group = lane >> 3, sub = lane & 7;
    for (int m = 0; m < M; ++m) {
        const int k = lane + 32 * m;
        bool open = k < n_sphere && !((buried >> m) & 1u);
        if (open) {
            const float3 p = sphere_point(A, a, dirs, k);
            for (int t = 0; t < n_near; ++t)
                if (inside(p, nb[t])) {
                    buried |= 1u << m;
                    open = false;
                    break;
                }
        }
        for (unsigned left = __ballot_sync(0xffffffffu, open); left;) {
            int b = -1;                                  // this group's point: the group-th one left
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (group == q && left) b = __ffs(left) - 1;
                left &= left - 1;                        // stays 0 once it is
            }
            bool hit = false;
            if (b >= 0) {
                const float3 p = sphere_point(A, a, dirs, b + 32 * m);
                for (int t = sub; t < n_far && !hit; t += 8) hit = inside(p, nb[kNb - 1 - t]);
            }
            // the points found inside, as bits of the lanes that own them
            const unsigned hits = __ballot_sync(0xffffffffu, hit);
            const bool found = b >= 0 && ((hits >> (8 * group)) & 0xffu);
            const unsigned mine = __reduce_or_sync(0xffffffffu, found ? 1u << b : 0u);
            if ((mine >> lane) & 1u) buried |= 1u << m;
        }
    }
    return buried;
}

// Issue-bound: 100 lattice points per atom against the 57 spheres that can reach them. A warp that
// tested the spheres in cell order, lanes waiting for the slowest, took 36 us for 8,000 atoms (22 of 32
// lanes active) and 195 us for seven receptors of 36,700 atoms in all, one after another; these take 75 us in
// one launch, 16 instead of 23 us for 1,500 atoms. Near spheres: closer than 1.1 a, about a dozen.
__global__ void __launch_bounds__(kSasWarps * 32) sas_kernel(const SurfaceItem* __restrict__ items,
                                                             const float* __restrict__ dirs, int n_sphere) {
    __shared__ float4 s_nb[kSasWarps][kNb];
    const SurfaceItem& g = items[blockIdx.y];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int s = blockIdx.x * kSasWarps + wib;
    if (s >= g.n) return;                               // warp-uniform
    float4* nb = s_nb[wib];
    const float4* sorted = g.sorted;
    const float* srad = g.srad;
    const float4 A = sorted[s];
    const float a = srad[s];
    const float reach = a + g.reach_max;
    const AtomGrid G = g.G;
    int c0[3], c1[3];
    const float pa[3] = {A.x, A.y, A.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c0[k] = cell_coord(pa[k] - reach, G.lo[k], G.inv_cell, G.cd[k]);
        c1[k] = cell_coord(pa[k] + reach, G.lo[k], G.inv_cell, G.cd[k]);
    }
    const float near2 = 1.2f * a * a;
    const float slack = 1e-2f + 1e-6f * (fabsf(A.x) + fabsf(A.y) + fabsf(A.z));
    uint32_t buried = 0;
    int n_near = 0, n_far = 0;
    // the rows of cells in reach, a lane each, 32 at a time; their atoms as one list
    const int ny = c1[1] - c0[1] + 1, n_rows = ny * (c1[2] - c0[2] + 1);
    for (int r0 = 0; r0 < n_rows; r0 += 32) {
        int b = 0, n = 0;
        if (r0 + lane < n_rows) {
            // the row's cells within reach of the atom (a little more than reach: cell borders are rounded)
            const int cz = c0[2] + (r0 + lane) / ny, cy = c0[1] + (r0 + lane) % ny;
            const float ylo = G.lo[1] + cy * kCell, zlo = G.lo[2] + cz * kCell;
            const float dy = fmaxf(0.f, fmaxf(ylo - A.y, A.y - (ylo + kCell)) - slack);
            const float dz = fmaxf(0.f, fmaxf(zlo - A.z, A.z - (zlo + kCell)) - slack);
            const float left = reach * reach - dy * dy - dz * dz;
            if (left > 0.f) {
                const float half = sqrtf(left) + slack;
                const int row = (cz * G.cd[1] + cy) * G.cd[0];
                b = g.cell_start[row + cell_coord(A.x - half, G.lo[0], G.inv_cell, G.cd[0])];
                n = g.cell_start[row + cell_coord(A.x + half, G.lo[0], G.inv_cell, G.cd[0]) + 1] - b;
            }
        }
        int end = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += y;
        }
        const int total = __shfl_sync(0xffffffffu, end, 31), shift = b - (end - n);
        for (int base = 0; base < total; base += 32) {
            const int p = base + lane;
            int row = 0;                                 // the rows that end at or before position p
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, end, row + o - 1) <= p) row += o;
            const int j = __shfl_sync(0xffffffffu, shift, row & 31) + p;
            bool take = false, near = false;
            float4 B = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p < total && j != s) {
                B = sorted[j];
                const float aj = srad[j];
                const float dx = B.x - A.x, dy = B.y - A.y, dz = B.z - A.z;
                const float lim = a + aj + 1e-3f;       // spheres that can overlap, with slack
                const float d2 = dx * dx + dy * dy + dz * dz;
                take = d2 < lim * lim;
                near = take && d2 < near2;
                B.w = aj * aj;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, take), baln = __ballot_sync(0xffffffffu, near);
            const unsigned below = (1u << lane) - 1u;
            if (near) nb[n_near + __popc(baln & below)] = B;
            else if (take) nb[kNb - 1 - (n_far + __popc(bal & ~baln & below))] = B;
            n_near += __popc(baln);
            n_far += __popc(bal & ~baln);
            if (n_near + n_far > kNb - 32) {
                __syncwarp();
                buried = bury(nb, n_near, n_far, A, a, dirs, n_sphere, lane, buried);
                __syncwarp();
                n_near = n_far = 0;
            }
        }
    }
    __syncwarp();
    buried = bury(nb, n_near, n_far, A, a, dirs, n_sphere, lane, buried);
    const int M = (n_sphere + 31) >> 5;
    uint32_t valid = 0;
    for (int m = 0; m < M; ++m)
        if (lane + 32 * m < n_sphere) valid |= 1u << m;
    const uint32_t keep = valid & ~buried;
    const int i = __float_as_int(A.w);
    g.kept[(size_t)i * 32 + lane] = keep;
    const int c = __reduce_add_sync(0xffffffffu, __popc(keep));
    if (lane == 0) g.n_kept[i] = c;
}

// First points of the atoms, in input order (blockIdx.x 0) and in cell order (1).
__global__ void __launch_bounds__(1024) point_scan_kernel(const SurfaceItem* __restrict__ items) {
    const SurfaceItem& g = items[blockIdx.y];
    const int *n_kept = g.n_kept, *order = g.order;
    if (blockIdx.x == 0) {
        const int total = block_scan([&](int i) { return n_kept[i]; }, g.n, g.offset);
        if (threadIdx.x == 0) g.status[1] = total;
    } else {
        block_scan([&](int i) { return n_kept[order[i]]; }, g.n, g.offset_sorted);
    }
}

// Kept points in (atom, k) order, a warp per atom, and their grouping by the cell order of the atoms.
__global__ void __launch_bounds__(128) sas_write_kernel(const SurfaceItem* __restrict__ items,
                                                        const float* __restrict__ dirs, int n_sphere) {
    const SurfaceItem& g = items[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const int s = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (s >= g.n) return;
    const int i = g.order[s];
    const float4 A = g.atoms[i];
    const float a = g.arad[i];
    const uint32_t word = g.kept[(size_t)i * 32 + lane];
    int base = g.offset[i];
    const int shift = g.offset_sorted[s] - base;
    const int M = (n_sphere + 31) >> 5;
    for (int m = 0; m < M; ++m) {
        const bool on = (word >> m) & 1u;
        const unsigned bal = __ballot_sync(0xffffffffu, on);
        if (on) {
            const int k = lane + 32 * m;
            const int pos = base + __popc(bal & ((1u << lane) - 1u));
            const float3 p = sphere_point(A, a, dirs, k);
            g.pts[3 * (size_t)pos] = p.x;
            g.pts[3 * (size_t)pos + 1] = p.y;
            g.pts[3 * (size_t)pos + 2] = p.z;
            g.src[pos] = i * n_sphere + k;
            g.perm[pos + shift] = pos;
        }
        base += __popc(bal);
    }
}

// ------------------------------------------------------------ Step 2: Eq. 1 + protrusion ---

struct FeatArgs {
    const float4* sorted;
    const int* cell_start;
    AtomGrid G;
    const float* pts;
    const int* perm;         // [n_pts] order in which points are grouped, or null (given order)
    int n_pts;
    const float* props;      // [n_atoms][n_props], input atom order
    int n_props;
    float inv_rf, rf2, rp2, reach, reach_f;   // reach: of either radius, reach_f: of the features
    float* feat;             // [n_pts][n_props]
    int* prot;               // [n_pts] or null
};

// The smallest of a warp's values, through the integer reduction on an order-preserving image.
__device__ __forceinline__ float warp_min(float v) {
    int i = __float_as_int(v);
    i = __reduce_min_sync(0xffffffffu, i ^ ((i >> 31) & 0x7fffffff));
    return __int_as_float(i ^ ((i >> 31) & 0x7fffffff));
}

// One CTA per group of 32 points. The cell rows within reach of the group's bounding box (each
// row's x range trimmed to the box swept by the reach) are listed with their atom counts, up to
// kFeatRows at a time, and the concatenated atoms of the listed rows are cut into chunks of 32:
// the CTA's kFeatSplit warps take the chunks in turn (balanced to within one chunk), each loading
// its next chunk into registers while it works on the current one, keeping of a chunk the atoms within
// reach of the box (about half), those within the feature radius of it first, and testing two atoms at a
// time in packed arithmetic; the partial sums are added in shared memory at the end.
//
// Bound by the latency of its phases at the warps that fit (registers): 12 warps by 3 CTAs per SM
// measured best, 36 us for 8,000 atoms with 7 columns and 63 us with 20 (event-timed), against 42 and 89 us
// for 16 warps by the 2 CTAs that 59 registers allow, 40 and 69 us for 8 warps by 4.
__global__ void __launch_bounds__(kFeatSplit * 32, 3) feature_kernel(FeatArgs g) {
    __shared__ __align__(16) float s_at[kFeatSplit][3][32];   // a chunk's atoms, read two at a time
    __shared__ float4 s_pr[kFeatSplit][32][kPropChunk / 4];   // an atom's chunk: two broadcast loads
    __shared__ float s_red[kFeatSplit][kPropChunk + 1][32];
    __shared__ int s_beg[kFeatRows];                          // first atom of a listed row
    __shared__ int s_off[kFeatRows + 1];                      // position of its atoms in the list
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int slot = blockIdx.x * 32 + lane;
    const int q0 = blockIdx.y * kPropChunk;
    const int nq = min(kPropChunk, g.n_props - q0);
    const bool live = slot < g.n_pts;
    const int pi = live ? (g.perm ? g.perm[slot] : slot) : 0;
    float px = 0.f, py = 0.f, pz = 0.f;
    if (live) {
        px = g.pts[3 * (size_t)pi];
        py = g.pts[3 * (size_t)pi + 1];
        pz = g.pts[3 * (size_t)pi + 2];
    }
    // the group's bounding box (non-finite points take no part); every warp computes the same one
    const bool fin = live && isfinite(px) && isfinite(py) && isfinite(pz);
    const float pos[3] = {px, py, pz};
    float lo3[3], hi3[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo3[k] = warp_min(fin ? pos[k] : INFINITY);
        hi3[k] = -warp_min(fin ? -pos[k] : INFINITY);
    }
    float acc[kPropChunk];
#pragma unroll
    for (int q = 0; q < kPropChunk; ++q) acc[q] = 0.f;
    int count = 0;
    if (lo3[0] <= hi3[0]) {                             // at least one finite point (CTA-uniform)
        const float reach2 = g.reach * g.reach, feat2 = g.reach_f * g.reach_f;
        const float cell = 1.0f / g.G.inv_cell;
        int c0[3], c1[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c0[k] = cell_coord(lo3[k] - g.reach, g.G.lo[k], g.G.inv_cell, g.G.cd[k]);
            c1[k] = cell_coord(hi3[k] + g.reach, g.G.lo[k], g.G.inv_cell, g.G.cd[k]);
        }
        const int ny = c1[1] - c0[1] + 1, n_rows = ny * (c1[2] - c0[2] + 1);
        for (int rbase = 0; rbase < n_rows; rbase += kFeatRows) {
            const int nr = min(kFeatRows, n_rows - rbase);
            // list the rows: begin and atom count (zero for a row out of reach)
            for (int t = threadIdx.x; t < nr; t += kFeatSplit * 32) {
                const int rr = rbase + t;
                const int cz = c0[2] + rr / ny, cy = c0[1] + rr % ny;
                const float ylo = g.G.lo[1] + cy * cell, zlo = g.G.lo[2] + cz * cell;
                const float dy = fmaxf(0.f, fmaxf(ylo - hi3[1], lo3[1] - (ylo + cell)));
                const float dz = fmaxf(0.f, fmaxf(zlo - hi3[2], lo3[2] - (zlo + cell)));
                const float dyz2 = dy * dy + dz * dz;
                int b = 0, n = 0;
                if (dyz2 <= reach2) {
                    const float half = sqrtf(reach2 - dyz2);
                    const int x0 = cell_coord(lo3[0] - half, g.G.lo[0], g.G.inv_cell, g.G.cd[0]);
                    const int x1 = cell_coord(hi3[0] + half, g.G.lo[0], g.G.inv_cell, g.G.cd[0]);
                    const int row = (cz * g.G.cd[1] + cy) * g.G.cd[0];
                    b = g.cell_start[row + x0];
                    n = g.cell_start[row + x1 + 1] - b;
                }
                s_beg[t] = b;
                s_off[t + 1] = n;
            }
            __syncthreads();
            if (wib == 0) {                             // prefix of the counts, 32 rows per pass
                int carry = 0;
                for (int t0 = 0; t0 < nr; t0 += 32) {
                    int v = t0 + lane < nr ? s_off[t0 + lane + 1] : 0;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, v, o);
                        if (lane >= o) v += y;
                    }
                    if (t0 + lane < nr) s_off[t0 + lane + 1] = carry + v;
                    carry += __shfl_sync(0xffffffffu, v, 31);
                }
                if (lane == 0) s_off[0] = 0;
            }
            __syncthreads();
            const int total = s_off[nr], n_chunks = (total + 31) >> 5;
            // the atom at list position p: its row by binary search over the offsets
            auto fetch = [&](int c, float4& B, int& kind, float (&v)[kPropChunk]) {
                const int p = c * 32 + lane;
                kind = 0;
                if (p < total) {
                    int lo = 0, hi = nr - 1;                // the last row with s_off[row] <= p
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (s_off[mid] <= p) lo = mid;
                        else hi = mid - 1;
                    }
                    B = g.sorted[s_beg[lo] + (p - s_off[lo])];
                    const float ex = fmaxf(0.f, fmaxf(lo3[0] - B.x, B.x - hi3[0])), ey = fmaxf(0.f, fmaxf(lo3[1] - B.y, B.y - hi3[1])),
                                ez = fmaxf(0.f, fmaxf(lo3[2] - B.z, B.z - hi3[2]));
                    const float e2 = ex * ex + ey * ey + ez * ez;
                    kind = e2 < feat2 ? 2 : (e2 < reach2 ? 1 : 0);
                    if (kind == 2) {
                        const float* pr = g.props + (size_t)__float_as_int(B.w) * g.n_props + q0;
#pragma unroll
                        for (int q = 0; q < kPropChunk; ++q) v[q] = q < nq ? __ldg(pr + q) : 0.f;
                    }
                }
            };
            float4 B_next = make_float4(0.f, 0.f, 0.f, 0.f);
            int kind_next = 0;
            float v_next[kPropChunk];
#pragma unroll
            for (int q = 0; q < kPropChunk; ++q) v_next[q] = 0.f;
            if (wib < n_chunks) fetch(wib, B_next, kind_next, v_next);
            for (int c = wib; c < n_chunks; c += kFeatSplit) {
                // the chunk's atoms in reach of the group's box, those within the feature radius of it first
                const unsigned in_f = __ballot_sync(0xffffffffu, kind_next == 2), in_r = __ballot_sync(0xffffffffu, kind_next == 1);
                const int nf = __popc(in_f), nt = nf + __popc(in_r);
                const unsigned below = (1u << lane) - 1u;
                __syncwarp();
                if (kind_next) {
                    const int at = kind_next == 2 ? __popc(in_f & below) : nf + __popc(in_r & below);
                    s_at[wib][0][at] = B_next.x;
                    s_at[wib][1][at] = B_next.y;
                    s_at[wib][2][at] = B_next.z;
                    if (kind_next == 2) {
#pragma unroll
                        for (int q = 0; q < kPropChunk / 4; ++q)
                            s_pr[wib][at][q] = make_float4(v_next[4 * q], v_next[4 * q + 1], v_next[4 * q + 2], v_next[4 * q + 3]);
                    }
                }
                if (lane < 3 && (nt & 1)) s_at[wib][lane][nt] = 1e15f;   // the last pair's second: beyond any radius
                __syncwarp();
                if (c + kFeatSplit < n_chunks) fetch(c + kFeatSplit, B_next, kind_next, v_next);
                auto pair_d2 = [&](int t) {                              // the chunk's atoms t and t + 1
                    const float2 ax = *reinterpret_cast<const float2*>(&s_at[wib][0][t]);
                    const float2 ay = *reinterpret_cast<const float2*>(&s_at[wib][1][t]);
                    const float2 az = *reinterpret_cast<const float2*>(&s_at[wib][2][t]);
                    const float2 dx = __fadd2_rn(ax, make_float2(-px, -px)), dy = __fadd2_rn(ay, make_float2(-py, -py)),
                                 dz = __fadd2_rn(az, make_float2(-pz, -pz));
                    const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)));
                    count += (d2.x <= g.rp2) + (d2.y <= g.rp2);
                    return d2;
                };
                int t = 0;
                for (; t < nf; t += 2) {
                    const float2 d2 = pair_d2(t);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float e = h ? d2.y : d2.x;
                        if (!(e < g.rf2)) continue;
                        const float w = 1.0f - sqrtf(e) * g.inv_rf;
#pragma unroll
                        for (int q = 0; q < kPropChunk / 4; ++q) {
                            const float4 pv = s_pr[wib][t + h][q];
                            acc[4 * q] = fmaf(w, pv.x, acc[4 * q]);
                            acc[4 * q + 1] = fmaf(w, pv.y, acc[4 * q + 1]);
                            acc[4 * q + 2] = fmaf(w, pv.z, acc[4 * q + 2]);
                            acc[4 * q + 3] = fmaf(w, pv.w, acc[4 * q + 3]);
                        }
                    }
                }
#pragma unroll 2
                for (; t < nt; t += 2) pair_d2(t);
            }
            __syncthreads();                            // the row table is rebuilt for the next rows
        }
    }
#pragma unroll
    for (int q = 0; q < kPropChunk; ++q) s_red[wib][q][lane] = acc[q];
    s_red[wib][kPropChunk][lane] = __int_as_float(count);
    __syncthreads();
    // the columns and the count are dealt to the warps, which all hold the same points
    if (!live) return;
    for (int q = wib; q < nq; q += kFeatSplit) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < kFeatSplit; ++w) v += s_red[w][q][lane];
        g.feat[(size_t)pi * g.n_props + q0 + q] = fin ? v : 0.f;
    }
    if (wib == kFeatSplit - 1 && g.prot && blockIdx.y == 0) {
        int total = 0;
#pragma unroll
        for (int w = 0; w < kFeatSplit; ++w) total += __float_as_int(s_red[w][kPropChunk][lane]);
        g.prot[pi] = fin ? total : 0;
    }
}

// ------------------------------------------------------------ Steps 4-5: clusters ---

// Spatial hash of a link-sized cell (Teschner et al., "Optimized Spatial Hashing for Collision
// Detection of Deformable Objects", VMV 2003).
__device__ __forceinline__ int cell_hash(int x, int y, int z, uint32_t mask) {
    return (int)((((uint32_t)x * 73856093u) ^ ((uint32_t)y * 19349663u) ^ ((uint32_t)z * 83492791u)) & mask);
}

// One point set of a clustering call (device pointers).
struct ClusterItem {
    const float* pts;
    const float* score;
    int n, n_buckets;
    float theta, link2, inv_cell;
    uint32_t hmask;
    int* key;                // [n] bucket of a clustered point, -1 otherwise
    int* count;              // [buckets] points of a bucket; counted down as they are placed
    int* start;              // [buckets + 1]
    float4* spts;            // clustered points in bucket order: (x, y, z, index bits)
    int* parent;             // [n]
    int* root;               // [n]
    int* cid;                // [n] cluster id of a root (order of discovery)
    double* s2;              // [n] per root
    double* sx;              // [n][3] per root
    int* size;               // [n] per root
    int* c_first;            // [n] root of a cluster id
    int* rank;               // [n] rank of a cluster id
    int* status;             // [0] error bits, [1] clusters
    int* cluster;            // [n] per point: its cluster's rank
    float* out;              // K clusters by rank: score [K], center [K][3], size [K], first [K]
};

__device__ __forceinline__ int3 link_cell(const float* p, float inv) {
    return make_int3(__float2int_rd(p[0] * inv), __float2int_rd(p[1] * inv), __float2int_rd(p[2] * inv));
}

__global__ void __launch_bounds__(256) cl_init_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    g.parent[i] = i;
    const float s = g.score[i];
    int k = -1;
    if (s >= g.theta) {
        const float* p = g.pts + 3 * (size_t)i;
        const float lim = 1073741824.0f;   // 2^30 cells
        bool ok = true;
#pragma unroll
        for (int c = 0; c < 3; ++c) ok = ok && isfinite(p[c]) && fabsf(p[c] * g.inv_cell) < lim;
        if (!ok) {
            atomicOr(g.status, kErrCoord);
        } else {
            const int3 c = link_cell(p, g.inv_cell);
            k = cell_hash(c.x, c.y, c.z, g.hmask);
            atomicAdd(&g.count[k], 1);
        }
    }
    g.key[i] = k;
}

__global__ void __launch_bounds__(1024) cl_scan_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int* count = g.count;
    block_scan([&](int i) { return count[i]; }, g.n_buckets, g.start);
}

// Clustered points into their buckets (in any order within one: nothing below depends on it): a
// neighbour scan reads each candidate with one contiguous load, and consecutive warps take
// neighbouring points.
__global__ void __launch_bounds__(256) cl_place_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    const int k = g.key[i];
    if (k < 0) return;
    const float* p = g.pts + 3 * (size_t)i;
    g.spts[g.start[k] + atomicSub(&g.count[k], 1) - 1] = make_float4(p[0], p[1], p[2], __int_as_float(i));
}

// Root of v: parents only ever point to lower indices, so the walk ends.
__device__ __forceinline__ int uf_find(int* par, int v) {
    int cur = __ldcg(par + v);
    if (cur != v) {
        int prev = v, next;
        while (cur > (next = __ldcg(par + cur))) {   // path halving towards the root
            par[prev] = next;
            prev = cur;
            cur = next;
        }
    }
    return cur;
}

// Joins the components of a and b, hooking the larger root under the smaller. Every failed
// attempt lowers a + b, so the loop ends; the bound only guards against a broken invariant.
__device__ __forceinline__ bool uf_unite(int* par, int a, int b) {
    a = uf_find(par, a);
    b = uf_find(par, b);
    for (int it = 0; it < (1 << 26) && a != b; ++it) {
        if (a > b) { const int t = a; a = b; b = t; }
        const int old = atomicCAS(par + b, b, a);
        if (old == b) return true;
        b = uf_find(par, old);
        a = uf_find(par, a);
    }
    return a == b;
}

// One warp per clustered point: lane l < 27 scans link cell l of the 27 around q's cell and calls
// f(j) for every clustered point j within the link of q there (q included; two cells that share a
// hash bucket are scanned twice, which changes nothing below).
template <typename F>
__device__ __forceinline__ void for_linked_lane(const ClusterItem& g, const float4& q, int lane, F&& f) {
    if (lane >= 27) return;
    const float p3[3] = {q.x, q.y, q.z};
    const int3 c = link_cell(p3, g.inv_cell);
    const int h = cell_hash(c.x + lane % 3 - 1, c.y + (lane / 3) % 3 - 1, c.z + lane / 9 - 1, g.hmask);
    const float4* spts = g.spts;
    const float link2 = g.link2;
    const int e = g.start[h + 1];
    for (int u = g.start[h]; u < e; ++u) {
        const float4 o = spts[u];
        const float ex = o.x - q.x, ey = o.y - q.y, ez = o.z - q.z;
        if (ex * ex + ey * ey + ez * ez <= link2) f(__float_as_int(o.w));
    }
}

// One hooking round: every clustered point takes the lowest parent among its linked points and
// lowers its own tree's root to it (atomicMin keeps parent[x] <= x, and every hook follows a
// link, so trees only ever join points of one component). From parent[i] = i the first round
// builds a shallow forest (each point under its lowest-index linked point); after a flattening
// pass each further round joins neighbouring trees, so their number falls quickly and the
// lock-free unions that follow have little left to do.
__global__ void __launch_bounds__(256) cl_hook_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= g.start[g.n_buckets]) return;              // warp-uniform
    const float4 q = g.spts[w];
    int* parent = g.parent;
    const int ri = __ldcg(parent + __float_as_int(q.w));
    int m = ri;
    for_linked_lane(g, q, lane, [&](int j) { m = min(m, __ldcg(parent + j)); });
    m = __reduce_min_sync(0xffffffffu, m);
    if (lane == 0 && m < ri) atomicMin(parent + ri, m);
}

// Points every clustered point at the root of its tree (each thread writes only its own entry;
// a concurrent write elsewhere only shortens the walk), so that most linked pairs are seen to
// share a tree by one comparison.
__global__ void __launch_bounds__(256) cl_flatten_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.start[g.n_buckets]) return;
    const int i = __float_as_int(g.spts[t].w);
    int* parent = g.parent;
    int r = __ldcg(parent + i);
    for (int next; (next = __ldcg(parent + r)) < r;) r = next;
    parent[i] = r;
}

__global__ void __launch_bounds__(256) cl_union_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= g.start[g.n_buckets]) return;              // warp-uniform
    const float4 q = g.spts[w];
    const int i = __float_as_int(q.w);
    int* parent = g.parent;
    bool ok = true;
    for_linked_lane(g, q, lane, [&](int j) {
        // components only ever merge, so equal parents mean the pair is already joined
        if (j > i && __ldcg(parent + i) != __ldcg(parent + j)) ok = uf_unite(parent, i, j) && ok;
    });
    if (!ok) atomicOr(g.status, kErrUnion);
}

// Roots, cluster ids (from a counter, so in any order: everything below depends only on the ranking,
// which is unique) and the sums of each cluster in float64.
__global__ void __launch_bounds__(256) cl_stats_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    const int r = g.key[i] < 0 ? -1 : uf_find(g.parent, i);
    g.root[i] = r;
    if (r == i) {
        const int c = atomicAdd(g.status + 1, 1);
        g.cid[i] = c;
        g.c_first[c] = i;
    }
    if (r < 0) return;
    const double s = g.score[i];
    atomicAdd(g.s2 + r, s * s);
    for (int c = 0; c < 3; ++c) atomicAdd(g.sx + 3 * (size_t)r + c, (double)g.pts[3 * (size_t)i + c]);
    atomicAdd(g.size + r, 1);
}

// rank of cluster c = the number of clusters sorting before it (score desc, first index asc)
__global__ void __launch_bounds__(256) cl_rank_kernel(const ClusterItem* __restrict__ items) {
    __shared__ double s_s[256];
    __shared__ int s_f[256];
    const ClusterItem& g = items[blockIdx.y];
    const int K = g.status[1];
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if ((int)(blockIdx.x * blockDim.x) >= K) return;    // block-uniform
    const int fc = c < K ? g.c_first[c] : 0;
    const double sc = c < K ? g.s2[fc] : 0.0;
    int r = 0;
    for (int base = 0; base < K; base += 256) {
        __syncthreads();
        const int t = base + threadIdx.x;
        if (t < K) {
            const int f = g.c_first[t];
            s_f[threadIdx.x] = f;
            s_s[threadIdx.x] = g.s2[f];
        }
        __syncthreads();
        const int m = min(256, K - base);
        for (int u = 0; u < m; ++u) r += s_s[u] > sc || (s_s[u] == sc && s_f[u] < fc);
    }
    if (c < K) g.rank[c] = r;
}

__global__ void __launch_bounds__(256) cl_output_kernel(const ClusterItem* __restrict__ items) {
    const ClusterItem& g = items[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    const int r = g.root[i];
    g.cluster[i] = r < 0 ? -1 : g.rank[g.cid[r]];
    if (r != i) return;
    const int k = g.rank[g.cid[i]], m = g.size[i];
    const size_t K = (size_t)g.status[1];
    g.out[k] = (float)g.s2[i];
    for (int c = 0; c < 3; ++c) g.out[K + 3 * (size_t)k + c] = (float)(g.sx[3 * (size_t)i + c] / m);
    reinterpret_cast<int*>(g.out)[4 * K + k] = m;
    reinterpret_cast<int*>(g.out)[5 * K + k] = i;
}

// ------------------------------------------------------------------------- host side ---

// Device memory of the pocket side: one stream-ordered pool per device, owned by the library,
// that keeps freed blocks for reuse until the process exits (the device's default pool hands them
// back to the driver at every synchronisation, and mapping them again costs more than the
// kernels of a call).
cudaMemPool_t pocket_pool(int device, cudaError_t* err) {
    static std::mutex mu;
    static cudaMemPool_t pools[64] = {};
    if (device < 0 || device >= 64) {
        *err = cudaErrorInvalidDevice;
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[device]) {
        cudaMemPoolProps props;
        std::memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        cudaMemPool_t p = nullptr;
        *err = cudaMemPoolCreate(&p, &props);
        if (*err != cudaSuccess) return nullptr;
        uint64_t keep = ~0ull;
        *err = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (*err != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return nullptr;
        }
        pools[device] = p;
    }
    *err = cudaSuccess;
    return pools[device];
}

// The allocations of one object or one call, freed together in stream order.
struct Pool {
    cudaStream_t stream = nullptr;
    cudaMemPool_t mp = nullptr;
    std::vector<void*> ptrs;
    cudaError_t err = cudaSuccess;
    Pool() = default;
    Pool(cudaStream_t s, int device) { init(s, device); }
    void init(cudaStream_t s, int device) {
        stream = s;
        mp = pocket_pool(device, &err);
    }
    template <typename T>
    T* take(size_t count) {
        void* p = nullptr;
        if (err != cudaSuccess) return nullptr;
        err = cudaMallocFromPoolAsync(&p, count ? count * sizeof(T) : 16, mp, stream);
        if (err != cudaSuccess) return nullptr;
        ptrs.push_back(p);
        return (T*)p;
    }
    void release() {
        for (void* p : ptrs) cudaFreeAsync(p, stream);
        ptrs.clear();
    }
};

pv_status fail(pv_context* ctx, pv_status s, const char* msg) {
    pv::context_set_error(ctx, msg);
    return s;
}

pv_status cuda_fail(pv_context* ctx, cudaError_t e, const char* what) {
    static thread_local std::string m;
    m = std::string(what) + ": " + cudaGetErrorString(e);
    return fail(ctx, e == cudaErrorMemoryAllocation ? PV_ERR_OOM : PV_ERR_CUDA, m.c_str());
}

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetLastError();
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

bool valid_params(const pv_pocket_params* p) {
    return p && std::isfinite(p->probe) && p->probe >= 0.f && p->probe <= 10.f && p->n_sphere >= 1 &&
           p->n_sphere <= PV_MAX_SPHERE_POINTS && p->r_feature > 0.f && std::isfinite(p->r_feature) &&
           p->r_feature <= 100.f && p->r_protrusion > 0.f && p->r_protrusion <= 100.f &&
           std::isfinite(p->link) && p->link > 0.f && p->link <= 100.f && !std::isnan(p->threshold);
}

}  // namespace

struct pv_surface {
    int magic = kSurfaceMagic;
    pv_context* ctx = nullptr;
    int device = 0;
    Pool pool;
    int n_atoms = 0, n_points = 0, n_sphere = 0;
    AtomGrid G{};
    float4* sorted = nullptr;
    int* cell_start = nullptr;
    float* points = nullptr;
    int* src = nullptr;
    int* perm = nullptr;      // points grouped by the cell order of their atoms
};

struct pv_clusters {
    int magic = kClustersMagic;
    pv_context* ctx = nullptr;
    int device = 0;
    Pool pool;
    int n = 0, K = 0;
    int* data = nullptr;      // cluster [n], then score [K], center [K][3], size [K], first [K]
};

extern "C" pv_status pv_pocket_params_default(pv_pocket_params* p) {
    if (!p) return PV_ERR_ARG;
    p->probe = 1.6f;
    p->n_sphere = 100;
    p->r_feature = 6.0f;
    p->r_protrusion = 10.0f;
    p->threshold = 0.5f;
    p->link = 3.0f;
    return PV_OK;
}

namespace {

// Host and device memory laid out alike, filled on the host and uploaded by one copy.
struct Staging {
    std::vector<char> host;
    size_t take(size_t bytes) {
        const size_t at = (host.size() + 15) & ~(size_t)15;
        host.resize(at + bytes);
        return at;
    }
    size_t put(const void* p, size_t bytes) {
        const size_t at = take(bytes);
        std::memcpy(host.data() + at, p, bytes);
        return at;
    }
};

// Offsets of arrays in one allocation (256-byte aligned).
struct Carve {
    size_t bytes = 0;
    template <typename T>
    size_t take(size_t count) {
        const size_t at = (bytes + 255) & ~(size_t)255;
        bytes = at + count * sizeof(T);
        return at;
    }
};

// One receptor of a surface call on the host.
struct SurfaceJob {
    const pv_receptor* r = nullptr;
    const float* radius = nullptr;
    int n = 0;
    float r_max = 1.80f;
    AtomGrid G{};
    long long n_cells = 0;
    pv_surface* S = nullptr;
};

pv_status surface_check(pv_context* ctx, const SurfaceJob& J) {
    const pv_receptor* r = J.r;
    if (!r || r->n_atoms < 1 || r->n_atoms > kMaxAtoms) return fail(ctx, PV_ERR_ARG, "receptor atom count must be in [1, 200000]");
    if (!r->xyz || (!J.radius && !r->element)) return fail(ctx, PV_ERR_ARG, "receptor xyz and element (or radii) required");
    if (r->mem != PV_MEM_HOST && r->mem != PV_MEM_DEVICE) return fail(ctx, PV_ERR_ARG, "receptor mem kind");
    return PV_OK;
}

// The binning grid of a receptor from its bounding box.
pv_status surface_grid(pv_context* ctx, SurfaceJob& J, const double lo[3], const double hi[3]) {
    J.n_cells = 1;
    for (int k = 0; k < 3; ++k) {
        J.G.lo[k] = (float)(lo[k] - 0.5);
        J.G.cd[k] = (int)std::ceil((hi[k] + 0.5 - (double)J.G.lo[k]) / kCell) + 1;
        J.n_cells *= J.G.cd[k];
    }
    J.G.inv_cell = 1.0f / kCell;
    if (J.n_cells > (1 << 24)) return fail(ctx, PV_ERR_ARG, "receptor spans too large a region");
    return PV_OK;
}

// Validity and bounding box of every receptor: host arrays are read here, device-resident ones by one
// launch for all of them and one readback.
pv_status surface_prepare(pv_context* ctx, cudaStream_t st, int dev, std::vector<SurfaceJob>& jobs) {
    std::vector<BoundsItem> items;
    for (SurfaceJob& J : jobs) {
        const pv_status s = surface_check(ctx, J);
        if (s != PV_OK) return s;
        J.n = J.r->n_atoms;
        if (J.r->mem == PV_MEM_DEVICE) items.push_back(BoundsItem{J.r->xyz, J.radius, J.n});
    }
    std::vector<float> found(8 * items.size());
    if (!items.empty()) {
        Pool pool(st, dev);
        Carve c;
        const size_t o_items = c.take<BoundsItem>(items.size()), o_out = c.take<float>(found.size());
        char* d = pool.take<char>(c.bytes);
        cudaError_t e = pool.err;
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(d + o_items, items.data(), sizeof(BoundsItem) * items.size(), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) {
            bounds_kernel<<<(unsigned)items.size(), 1024, 0, st>>>((const BoundsItem*)(d + o_items), (float*)(d + o_out));
            e = cudaGetLastError();
        }
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(found.data(), d + o_out, sizeof(float) * found.size(), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        pool.release();
        if (e != cudaSuccess) return cuda_fail(ctx, e, "receptor read");
    }
    const float* f = found.data();
    for (SurfaceJob& J : jobs) {
        double lo[3] = {1e30, 1e30, 1e30}, hi[3] = {-1e30, -1e30, -1e30};
        bool bad_radius = false, bad_xyz = false;
        float r_max = 0.f;
        if (J.r->mem == PV_MEM_DEVICE) {
            int err;
            std::memcpy(&err, f + 7, sizeof(int));
            bad_radius = (err & kErrRadius) != 0;
            bad_xyz = (err & kErrCoord) != 0;
            for (int k = 0; k < 3; ++k) {
                lo[k] = f[k];
                hi[k] = f[3 + k];
            }
            r_max = f[6];
            f += 8;
        } else {
            const float* x = J.r->xyz;
            for (int i = 0; i < J.n; ++i)
                for (int k = 0; k < 3; ++k) {
                    const double v = x[3 * (size_t)i + k];
                    bad_xyz = bad_xyz || !(std::fabs(v) <= 1e6);
                    lo[k] = std::min(lo[k], v);
                    hi[k] = std::max(hi[k], v);
                }
            if (J.radius)
                for (int i = 0; i < J.n; ++i) {
                    bad_radius = bad_radius || !(J.radius[i] > 0.f && J.radius[i] <= 10.f);
                    r_max = std::max(r_max, J.radius[i]);
                }
        }
        if (bad_radius) return fail(ctx, PV_ERR_ARG, "atom radius must be in (0, 10] A");
        if (bad_xyz) return fail(ctx, PV_ERR_ARG, "receptor coordinates must be finite (|x| <= 1e6 A)");
        if (J.radius) J.r_max = r_max;   // bounds how far a neighbouring sphere can reach
        const pv_status s = surface_grid(ctx, J, lo, hi);
        if (s != PV_OK) return s;
    }
    return PV_OK;
}

// All receptors from their atoms to their points. The working memory of the call is one allocation;
// each surface keeps two (binned atoms; points). *bad: error bits found on the device.
cudaError_t surface_build(pv_context* ctx, cudaStream_t st, int dev, const pv_pocket_params* p,
                          std::vector<SurfaceJob>& jobs, Pool& scratch, int* bad, const char** stage) {
    const int k = (int)jobs.size(), ns = p->n_sphere;
    // lattice directions (spherical Fibonacci lattice, evaluated in double)
    std::vector<float> dirs(3 * (size_t)ns);
    const double golden_angle = kPi * (3.0 - std::sqrt(5.0));
    for (int j = 0; j < ns; ++j) {
        const double z = 1.0 - (2.0 * j + 1.0) / ns, rho = std::sqrt(std::max(0.0, 1.0 - z * z));
        dirs[3 * j] = (float)(rho * std::cos(golden_angle * j));
        dirs[3 * j + 1] = (float)(rho * std::sin(golden_angle * j));
        dirs[3 * j + 2] = (float)z;
    }
    // uploaded: records, directions, host receptors
    Staging up;
    const size_t o_items = up.take(sizeof(SurfaceItem) * k), o_dirs = up.put(dirs.data(), sizeof(float) * dirs.size());
    std::vector<size_t> o_xyz(k), o_el(k), o_rad(k);
    Carve zero, work;        // cleared; written before it is read
    const size_t o_status = zero.take<int>(2 * (size_t)k);
    std::vector<size_t> o_count(k), o_head(k), o_atoms(k), o_arad(k), o_key(k), o_next(k), o_order(k), o_kept(k), o_nkept(k),
        o_off(k), o_offs(k);
    for (int j = 0; j < k; ++j) {
        const SurfaceJob& J = jobs[j];
        const size_t n = J.n;
        if (J.r->mem == PV_MEM_HOST) {
            o_xyz[j] = up.put(J.r->xyz, sizeof(float) * 3 * n);
            if (J.r->element && !J.radius) o_el[j] = up.put(J.r->element, n);
            if (J.radius) o_rad[j] = up.put(J.radius, sizeof(float) * n);
        }
        o_count[j] = zero.take<int>(J.n_cells);
        o_head[j] = zero.take<int>(J.n_cells);
        o_atoms[j] = work.take<float4>(n);
        o_arad[j] = work.take<float>(n);
        o_key[j] = work.take<int>(n);
        o_next[j] = work.take<int>(n);
        o_order[j] = work.take<int>(n);
        o_kept[j] = work.take<uint32_t>(32 * n);
        o_nkept[j] = work.take<int>(n);
        o_off[j] = work.take<int>(n + 1);
        o_offs[j] = work.take<int>(n + 1);
    }
    Carve all;
    const size_t a_up = all.take<char>(up.host.size()), a_zero = all.take<char>(zero.bytes), a_work = all.take<char>(work.bytes);
    *stage = "allocation";
    char* d = scratch.take<char>(all.bytes);
    if (!d) return scratch.err;
    char *d_up = d + a_up, *d_zero = d + a_zero, *d_work = d + a_work;
    std::vector<SurfaceItem> items(k);
    for (int j = 0; j < k; ++j) {
        SurfaceJob& J = jobs[j];
        const size_t n = J.n;
        pv_surface* S = J.S = new (std::nothrow) pv_surface();
        if (!S) return cudaErrorMemoryAllocation;
        S->ctx = ctx;
        S->device = dev;
        S->pool.init(st, dev);
        S->n_atoms = J.n;
        S->n_sphere = ns;
        S->G = J.G;
        Carve c;
        const size_t o_sorted = c.take<float4>(n), o_start = c.take<int>(J.n_cells + 1), o_srad = c.take<float>(n);
        char* keep = S->pool.take<char>(c.bytes);
        if (!keep) return S->pool.err;
        S->sorted = (float4*)(keep + o_sorted);
        S->cell_start = (int*)(keep + o_start);
        SurfaceItem& g = items[j];
        const bool host = J.r->mem == PV_MEM_HOST;
        g.xyz = host ? (const float*)(d_up + o_xyz[j]) : J.r->xyz;
        g.element = host ? (const uint8_t*)(d_up + o_el[j]) : J.r->element;
        g.radius = !J.radius ? nullptr : host ? (const float*)(d_up + o_rad[j]) : J.radius;
        g.n = J.n;
        g.n_cells = (int)J.n_cells;
        g.G = J.G;
        g.reach_max = J.r_max + p->probe + 1e-3f;
        g.atoms = (float4*)(d_work + o_atoms[j]);
        g.arad = (float*)(d_work + o_arad[j]);
        g.key = (int*)(d_work + o_key[j]);
        g.count = (int*)(d_zero + o_count[j]);
        g.head = (int*)(d_zero + o_head[j]);
        g.next = (int*)(d_work + o_next[j]);
        g.cell_start = S->cell_start;
        g.sorted = S->sorted;
        g.srad = (float*)(keep + o_srad);
        g.order = (int*)(d_work + o_order[j]);
        g.kept = (uint32_t*)(d_work + o_kept[j]);
        g.n_kept = (int*)(d_work + o_nkept[j]);
        g.offset = (int*)(d_work + o_off[j]);
        g.offset_sorted = (int*)(d_work + o_offs[j]);
        g.pts = nullptr;
        g.src = nullptr;
        g.perm = nullptr;
        g.status = (int*)(d_zero + o_status) + 2 * j;
    }
    std::memcpy(up.host.data() + o_items, items.data(), sizeof(SurfaceItem) * k);
    SurfaceItem* d_items = (SurfaceItem*)(d_up + o_items);
    const float* d_dirs = (const float*)(d_up + o_dirs);
    *stage = "receptor upload";
    cudaError_t e = cudaMemcpyAsync(d_up, up.host.data(), up.host.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_zero, 0, zero.bytes, st);
    if (e != cudaSuccess) return e;
    *stage = "surface points";
    auto extent = [&](int j) { return RunExtent{(jobs[j].n + kSasWarps - 1) / kSasWarps, 1}; };   // a warp per atom
    e = launch_runs(0, k, extent, [&](int y0, int ny, RunExtent most) {
        const unsigned bw = (unsigned)most.x, b256 = (bw * kSasWarps + 255) / 256;
        const SurfaceItem* it = d_items + y0;
        prep_atoms_kernel<<<dim3(b256, ny), 256, 0, st>>>(it, p->probe);
        cell_scan_kernel<<<dim3(1, ny), 1024, 0, st>>>(it);
        sort_atoms_kernel<<<dim3(b256, ny), 256, 0, st>>>(it);
        sas_kernel<<<dim3(bw, ny), kSasWarps * 32, 0, st>>>(it, d_dirs, ns);
        point_scan_kernel<<<dim3(2, ny), 1024, 0, st>>>(it);
        return cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    // one readback of all error words and point counts
    *stage = "readback";
    std::vector<int> status(2 * (size_t)k, 0);
    e = cudaMemcpyAsync(status.data(), d_zero + o_status, sizeof(int) * status.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    for (int j = 0; j < k; ++j) *bad |= status[2 * j];
    if (*bad) return cudaSuccess;
    // the points, their sources and the order in which the feature kernel groups them
    *stage = "point allocation";
    for (int j = 0; j < k; ++j) {
        pv_surface* S = jobs[j].S;
        S->n_points = status[2 * j + 1];
        const size_t m = S->n_points > 0 ? S->n_points : 1;
        Carve c;
        const size_t o_pts = c.take<float>(3 * m), o_src = c.take<int>(m), o_perm = c.take<int>(m);
        char* keep = S->pool.take<char>(c.bytes);
        if (!keep) return S->pool.err;
        items[j].pts = S->points = (float*)(keep + o_pts);
        items[j].src = S->src = (int*)(keep + o_src);
        items[j].perm = S->perm = (int*)(keep + o_perm);
    }
    *stage = "point order";
    e = cudaMemcpyAsync(d_items, items.data(), sizeof(SurfaceItem) * k, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    e = launch_runs(0, k, extent, [&](int y0, int ny, RunExtent most) {
        static_assert(kSasWarps == 4, "sas_write_kernel takes four atoms per block");
        sas_write_kernel<<<dim3((unsigned)most.x, ny), 128, 0, st>>>(d_items + y0, d_dirs, ns);
        return cudaGetLastError();
    });
    return e;
}

}  // namespace

extern "C" pv_status pv_surface_create_many(pv_context* ctx, int32_t n_receptors, const pv_receptor* receptors,
                                            const float* const* radii, const pv_pocket_params* p, pv_surface** out) {
    int dev = 0;
    cudaStream_t st = nullptr;
    if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
    if (!out || n_receptors < 1 || !receptors) return fail(ctx, PV_ERR_ARG, "receptors and out required");
    for (int j = 0; j < n_receptors; ++j) out[j] = nullptr;
    if (!valid_params(p)) return fail(ctx, PV_ERR_ARG, "pocket parameters out of range");
    DeviceGuard guard(dev);
    std::vector<SurfaceJob> jobs(n_receptors);
    for (int j = 0; j < n_receptors; ++j) {
        jobs[j].r = receptors + j;
        jobs[j].radius = radii ? radii[j] : nullptr;
    }
    const pv_status ps = surface_prepare(ctx, st, dev, jobs);
    if (ps != PV_OK) return ps;
    Pool scratch(st, dev);
    int bad = 0;
    const char* stage = "allocation";
    cudaError_t e = scratch.err;
    if (e == cudaSuccess) e = surface_build(ctx, st, dev, p, jobs, scratch, &bad, &stage);
    scratch.release();   // stream-ordered: after the kernels above
    if (e != cudaSuccess || bad) {
        for (SurfaceJob& J : jobs)
            if (J.S) {
                J.S->pool.release();
                delete J.S;
            }
        if (e != cudaSuccess) return cuda_fail(ctx, e, (std::string("surface: ") + stage).c_str());
        return fail(ctx, PV_ERR_ARG, (bad & kErrElement) ? "receptor element must be 0..3"
                                     : (bad & kErrRadius) ? "atom radius must be in (0, 10] A"
                                                          : "receptor coordinates must be finite");
    }
    for (int j = 0; j < n_receptors; ++j) out[j] = jobs[j].S;
    return PV_OK;
}

extern "C" pv_status pv_surface_create(pv_context* ctx, const pv_receptor* r, const float* radius,
                                       const pv_pocket_params* p, pv_surface** out) {
    if (!out) {
        int dev = 0;
        cudaStream_t st = nullptr;
        if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
        return fail(ctx, PV_ERR_ARG, "out is null");
    }
    *out = nullptr;
    if (!r) {
        int dev = 0;
        cudaStream_t st = nullptr;
        if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
        return fail(ctx, PV_ERR_ARG, "receptor atom count must be in [1, 200000]");
    }
    return pv_surface_create_many(ctx, 1, r, radius ? &radius : nullptr, p, out);
}

extern "C" pv_status pv_surface_info(const pv_surface* s, int32_t* n_atoms, int32_t* n_points) {
    if (!s || s->magic != kSurfaceMagic) return PV_ERR_STATE;
    if (n_atoms) *n_atoms = s->n_atoms;
    if (n_points) *n_points = s->n_points;
    return PV_OK;
}

extern "C" pv_status pv_surface_points(const pv_surface* s, const float** dev_xyz) {
    if (!s || s->magic != kSurfaceMagic) return PV_ERR_STATE;
    if (!dev_xyz) return PV_ERR_ARG;
    *dev_xyz = s->points;
    return PV_OK;
}

extern "C" pv_status pv_surface_read(pv_context* ctx, const pv_surface* s, float* xyz, int32_t* src, int32_t mem) {
    int dev = 0;
    cudaStream_t st = nullptr;
    if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
    if (!s || s->magic != kSurfaceMagic || s->ctx != ctx) return fail(ctx, PV_ERR_STATE, "surface of another context");
    if (mem != PV_MEM_HOST && mem != PV_MEM_DEVICE) return fail(ctx, PV_ERR_ARG, "mem kind");
    DeviceGuard guard(dev);
    const cudaMemcpyKind kind = mem == PV_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    cudaError_t e = cudaSuccess;
    if (s->n_points > 0 && xyz) e = cudaMemcpyAsync(xyz, s->points, sizeof(float) * 3 * s->n_points, kind, st);
    if (e == cudaSuccess && s->n_points > 0 && src) e = cudaMemcpyAsync(src, s->src, sizeof(int) * s->n_points, kind, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? PV_OK : cuda_fail(ctx, e, "surface read");
}

extern "C" pv_status pv_surface_features(pv_context* ctx, const pv_surface* s, int32_t n_points,
                                         const float* xyz, int32_t xyz_mem, int32_t n_props,
                                         const float* props, int32_t props_mem, const pv_pocket_params* p,
                                         float* dev_features, int32_t* dev_protrusion) {
    int dev = 0;
    cudaStream_t st = nullptr;
    if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
    if (!s || s->magic != kSurfaceMagic || s->ctx != ctx) return fail(ctx, PV_ERR_STATE, "surface of another context");
    if (!valid_params(p)) return fail(ctx, PV_ERR_ARG, "pocket parameters out of range");
    if (n_points < 0 || (!xyz && n_points != s->n_points)) return fail(ctx, PV_ERR_ARG, "n_points must equal the surface's count when xyz is NULL");
    if (n_props < 1 || n_props > PV_MAX_PROPS || !props) return fail(ctx, PV_ERR_ARG, "1..64 property columns required");
    if ((xyz && xyz_mem != PV_MEM_HOST && xyz_mem != PV_MEM_DEVICE) || (props_mem != PV_MEM_HOST && props_mem != PV_MEM_DEVICE))
        return fail(ctx, PV_ERR_ARG, "mem kind");
    if (n_points > 0 && !dev_features) return fail(ctx, PV_ERR_ARG, "dev_features is null");
    if (n_points == 0) return PV_OK;
    DeviceGuard guard(dev);
    Pool scratch(st, dev);
    const float* d_pts = xyz ? xyz : s->points;
    const float* d_props = props;
    cudaError_t e = cudaSuccess;
    if (xyz && xyz_mem == PV_MEM_HOST) {
        float* t = scratch.take<float>(3 * (size_t)n_points);
        if (t) e = cudaMemcpyAsync(t, xyz, sizeof(float) * 3 * (size_t)n_points, cudaMemcpyHostToDevice, st);
        d_pts = t;
    }
    if (props_mem == PV_MEM_HOST) {
        float* t = scratch.take<float>((size_t)s->n_atoms * n_props);
        if (t && e == cudaSuccess)
            e = cudaMemcpyAsync(t, props, sizeof(float) * (size_t)s->n_atoms * n_props, cudaMemcpyHostToDevice, st);
        d_props = t;
    }
    if (scratch.err != cudaSuccess) e = scratch.err;
    if (e == cudaSuccess) {
        FeatArgs a;
        a.sorted = s->sorted;
        a.cell_start = s->cell_start;
        a.G = s->G;
        a.pts = d_pts;
        a.perm = xyz ? nullptr : s->perm;
        a.n_pts = n_points;
        a.props = d_props;
        a.n_props = n_props;
        a.inv_rf = (float)(1.0 / (double)p->r_feature);
        a.rf2 = p->r_feature * p->r_feature;
        a.rp2 = p->r_protrusion * p->r_protrusion;
        a.reach = std::max(p->r_feature, p->r_protrusion) + 1e-3f;
        a.reach_f = p->r_feature + 1e-3f;
        a.feat = dev_features;
        a.prot = dev_protrusion;
        const dim3 grid((unsigned)((n_points + 31) / 32), (unsigned)((n_props + kPropChunk - 1) / kPropChunk));
        feature_kernel<<<grid, kFeatSplit * 32, 0, st>>>(a);
        e = cudaGetLastError();
    }
    scratch.release();   // stream-ordered: the kernel above finishes first
    return e == cudaSuccess ? PV_OK : cuda_fail(ctx, e, "surface features");
}

extern "C" void pv_surface_destroy(pv_surface* s) {
    if (!s || s->magic != kSurfaceMagic) return;
    DeviceGuard guard(s->device);
    s->pool.release();
    s->magic = 0;
    delete s;
}

namespace {

// Steps 4-5 for all point sets, issued on the stream; status[2 j], status[2 j + 1] (host) receive the
// error word and the cluster count of set j.
cudaError_t cluster_build(pv_context* ctx, cudaStream_t st, int dev, int k, const int32_t* n_points,
                          const float* const* dev_xyz, const float* const* dev_score, const pv_pocket_params* p,
                          std::vector<pv_clusters*>& cs, Pool& scratch, std::vector<int>& status, const char** stage) {
    *stage = "allocation";
    Carve zero, work;        // cleared; written before it is read
    const size_t o_items = work.take<ClusterItem>(k), o_status = zero.take<int>(2 * (size_t)k);
    std::vector<ClusterItem> items(k);
    // two passes over the same layout: offsets first, then addresses in the one allocation
    char *d_zero = nullptr, *d_work = nullptr;
    for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
            Carve all;
            const size_t a_zero = all.take<char>(zero.bytes), a_work = all.take<char>(work.bytes);
            char* d = scratch.take<char>(all.bytes);
            if (!d) return scratch.err;
            d_zero = d + a_zero;
            d_work = d + a_work;
            zero = Carve();
            work = Carve();
            work.take<ClusterItem>(k);
            zero.take<int>(2 * (size_t)k);
        }
        for (int j = 0; j < k; ++j) {
            const size_t m = n_points[j] > 0 ? n_points[j] : 1;
            uint32_t buckets = 1024;
            while (2 * buckets < (uint32_t)n_points[j]) buckets <<= 1;
            ClusterItem& g = items[j];
            g.n = n_points[j];
            g.n_buckets = (int)buckets;
            g.hmask = buckets - 1;
            g.count = (int*)(d_zero + zero.take<int>(buckets));
            g.s2 = (double*)(d_zero + zero.take<double>(m));
            g.sx = (double*)(d_zero + zero.take<double>(3 * m));
            g.size = (int*)(d_zero + zero.take<int>(m));
            g.start = (int*)(d_work + work.take<int>(buckets + 1));
            g.key = (int*)(d_work + work.take<int>(m));
            g.spts = (float4*)(d_work + work.take<float4>(m));
            g.parent = (int*)(d_work + work.take<int>(m));
            g.root = (int*)(d_work + work.take<int>(m));
            g.cid = (int*)(d_work + work.take<int>(m));
            g.c_first = (int*)(d_work + work.take<int>(m));
            g.rank = (int*)(d_work + work.take<int>(m));
        }
    }
    for (int j = 0; j < k; ++j) {
        pv_clusters* C = cs[j] = new (std::nothrow) pv_clusters();
        if (!C) return cudaErrorMemoryAllocation;
        C->ctx = ctx;
        C->device = dev;
        C->pool.init(st, dev);
        C->n = n_points[j];
        C->data = C->pool.take<int>(7 * (size_t)(C->n > 0 ? C->n : 1));
        if (!C->data) return C->pool.err;
        ClusterItem& g = items[j];
        g.pts = dev_xyz[j];
        g.score = dev_score[j];
        g.theta = p->threshold;
        g.link2 = p->link * p->link;
        // cells a little wider than the link so that linked points always sit in adjacent cells
        g.inv_cell = (float)(1.0 / ((double)p->link * (1.0 + 1e-5)));
        g.status = (int*)(d_zero + o_status) + 2 * j;
        g.cluster = C->data;
        g.out = (float*)(C->data + C->n);
    }
    *stage = "memset";
    cudaError_t e = cudaMemcpyAsync(d_work + o_items, items.data(), sizeof(ClusterItem) * k, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_zero, 0, zero.bytes, st);
    if (e != cudaSuccess) return e;
    *stage = "single linkage";
    // a warp per point in most kernels, 8 points per block
    e = launch_runs(0, k, [&](int j) { return RunExtent{((long long)n_points[j] + 7) / 8, 1}; }, [&](int y0, int ny, RunExtent most) {
        const unsigned bw = (unsigned)most.x, b = (bw * 8 + 255) / 256;
        const ClusterItem* it = (const ClusterItem*)(d_work + o_items) + y0;
        cl_init_kernel<<<dim3(b, ny), 256, 0, st>>>(it);
        cl_scan_kernel<<<dim3(1, ny), 1024, 0, st>>>(it);
        cl_place_kernel<<<dim3(b, ny), 256, 0, st>>>(it);
        for (int round = 0; round < kHookRounds; ++round) {
            cl_hook_kernel<<<dim3(bw, ny), 256, 0, st>>>(it);
            cl_flatten_kernel<<<dim3(b, ny), 256, 0, st>>>(it);
        }
        cl_union_kernel<<<dim3(bw, ny), 256, 0, st>>>(it);
        cl_stats_kernel<<<dim3(b, ny), 256, 0, st>>>(it);
        cl_rank_kernel<<<dim3(b, ny), 256, 0, st>>>(it);
        cl_output_kernel<<<dim3(b, ny), 256, 0, st>>>(it);
        return cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    // one readback of all error words and cluster counts
    *stage = "readback";
    e = cudaMemcpyAsync(status.data(), d_zero + o_status, sizeof(int) * status.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
}

}  // namespace

extern "C" pv_status pv_cluster_points_many(pv_context* ctx, int32_t n_sets, const int32_t* n_points,
                                            const float* const* dev_xyz, const float* const* dev_score,
                                            const pv_pocket_params* p, pv_clusters** out) {
    int dev = 0;
    cudaStream_t st = nullptr;
    if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
    if (!out || n_sets < 1 || !n_points || !dev_xyz || !dev_score) return fail(ctx, PV_ERR_ARG, "point sets and out required");
    for (int j = 0; j < n_sets; ++j) out[j] = nullptr;
    if (!valid_params(p)) return fail(ctx, PV_ERR_ARG, "pocket parameters out of range");
    for (int j = 0; j < n_sets; ++j) {
        if (n_points[j] < 0 || n_points[j] > (1 << 26)) return fail(ctx, PV_ERR_ARG, "point count must be in [0, 2^26]");
        if (n_points[j] > 0 && (!dev_xyz[j] || !dev_score[j])) return fail(ctx, PV_ERR_ARG, "dev_xyz and dev_score required");
    }
    DeviceGuard guard(dev);
    std::vector<pv_clusters*> cs(n_sets, nullptr);
    auto release_all = [&]() {
        for (pv_clusters*& C : cs)
            if (C) {
                C->pool.release();
                delete C;
                C = nullptr;
            }
    };
    Pool scratch(st, dev);
    std::vector<int> h_status(2 * (size_t)n_sets, 0);
    cudaError_t e = scratch.err;
    const char* stage = "allocation";
    if (e == cudaSuccess)
        e = cluster_build(ctx, st, dev, n_sets, n_points, dev_xyz, dev_score, p, cs, scratch, h_status, &stage);
    scratch.release();   // stream-ordered: after the kernels above
    if (e != cudaSuccess) {
        release_all();
        return cuda_fail(ctx, e, (std::string("clusters: ") + stage).c_str());
    }
    int bad = 0;
    for (int j = 0; j < n_sets; ++j) bad |= h_status[2 * j];
    if (bad) {
        release_all();
        return fail(ctx, PV_ERR_ARG, (bad & kErrCoord) ? "clustered points need finite coordinates within 2^30 link lengths"
                                                       : "union-find did not converge");
    }
    for (int j = 0; j < n_sets; ++j) {
        cs[j]->K = h_status[2 * j + 1];
        out[j] = cs[j];
    }
    return PV_OK;
}

extern "C" pv_status pv_cluster_points(pv_context* ctx, int32_t n, const float* dev_xyz, const float* dev_score,
                                       const pv_pocket_params* p, pv_clusters** out) {
    if (!out) {
        int dev = 0;
        cudaStream_t st = nullptr;
        if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
        return fail(ctx, PV_ERR_ARG, "out is null");
    }
    return pv_cluster_points_many(ctx, 1, &n, &dev_xyz, &dev_score, p, out);
}

extern "C" pv_status pv_clusters_info(const pv_clusters* c, int32_t* n_points, int32_t* n_clusters) {
    if (!c || c->magic != kClustersMagic) return PV_ERR_STATE;
    if (n_points) *n_points = c->n;
    if (n_clusters) *n_clusters = c->K;
    return PV_OK;
}

extern "C" pv_status pv_clusters_read(pv_context* ctx, const pv_clusters* c, int32_t* cluster, float* score,
                                      float* center, int32_t* size, int32_t* first, int32_t mem) {
    int dev = 0;
    cudaStream_t st = nullptr;
    if (!pv::context_device_stream(ctx, &dev, &st)) return PV_ERR_STATE;
    if (!c || c->magic != kClustersMagic || c->ctx != ctx) return fail(ctx, PV_ERR_STATE, "clusters of another context");
    if (mem != PV_MEM_HOST && mem != PV_MEM_DEVICE) return fail(ctx, PV_ERR_ARG, "mem kind");
    DeviceGuard guard(dev);
    const size_t n = (size_t)c->n, K = (size_t)c->K;
    const struct { void* dst; size_t at, count; } parts[5] = {
        {cluster, 0, n}, {score, n, K}, {center, n + K, 3 * K}, {size, n + 4 * K, K}, {first, n + 5 * K, K}};
    if (mem == PV_MEM_HOST) {   // one copy of the lot, without the points when they are not asked for
        const size_t from = cluster ? 0 : n;
        std::vector<int> all(n + 6 * K);
        cudaError_t e = all.size() == from ? cudaSuccess
                                           : cudaMemcpyAsync(all.data() + from, c->data + from,
                                                             sizeof(int) * (all.size() - from), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "clusters read");
        for (const auto& q : parts)
            if (q.dst && q.count) std::memcpy(q.dst, all.data() + q.at, sizeof(int) * q.count);
        return PV_OK;
    }
    cudaError_t e = cudaSuccess;
    for (const auto& q : parts)
        if (e == cudaSuccess && q.dst && q.count)
            e = cudaMemcpyAsync(q.dst, c->data + q.at, sizeof(int) * q.count, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? PV_OK : cuda_fail(ctx, e, "clusters read");
}

extern "C" void pv_clusters_destroy(pv_clusters* c) {
    if (!c || c->magic != kClustersMagic) return;
    DeviceGuard guard(c->device);
    c->pool.release();
    c->magic = 0;
    delete c;
}
