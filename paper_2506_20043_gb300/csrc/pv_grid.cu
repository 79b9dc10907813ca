// pv_grid.cu -- the grid cache ("Kernel 1", Methods "Accelerated Docking"; Supplementary
// Algorithm 2, Grid_cache(P)): receptor XS typing, binning of receptor atoms into cubic cells
// (CSR, deterministic order), and the map build. Each CTA owns a tile of 8 x 8 x 4 grid nodes and
// stages the receptor atoms within the cutoff of the tile's box (position, radius, flags) in shared memory;
// each of its warps walks those within the cutoff of its 4 x 4 x 4 nodes, and every lane accumulates, for two
// nodes, the Vina energy of each requested ligand XS type. Then the cell-packed copies of the maps.
#include "pv_internal.h"
#include "pv_runs.h"
#include "pv_device.cuh"

namespace pv {

constexpr int kTile = 8;             // nodes per tile edge along x and y
constexpr int kTileZ = 4;            // and along z
constexpr int kGridThreads = 32 * kTileZ;    // a warp per 4 x 4 x 4 nodes, two nodes per lane
constexpr int kMaxRows = 18;          // cells per axis within reach of a tile
constexpr int kStageCap = 768;       // staged receptor atoms per pass (about 200 are in a tile's reach)

__device__ __forceinline__ int xs_of(int el, int don, int acc, bool polar_c) {
    if (el == 0) return polar_c ? 1 : 0;
    if (el == 1) return 2 + (don ? 1 : 0) + (acc ? 2 : 0);
    if (el == 2) return 6 + (don ? 1 : 0) + (acc ? 2 : 0);
    return 10;
}

__device__ __forceinline__ int cell_index(float4 p, const float* lo, float inv_cell, const int* cd) {
    int cx = (int)floorf((p.x - lo[0]) * inv_cell);
    int cy = (int)floorf((p.y - lo[1]) * inv_cell);
    int cz = (int)floorf((p.z - lo[2]) * inv_cell);
    if (cx < 0 || cy < 0 || cz < 0 || cx >= cd[0] || cy >= cd[1] || cz >= cd[2]) return -1;
    return (cz * cd[1] + cy) * cd[0] + cx;
}

struct CellGrid {
    float lo[3];
    float inv_cell;
    int cd[3];
};

// Typing and binning of receptor atoms, O(n) and without a host round trip. Typing needs the N and O
// within 1.75 A of a carbon, binning a stable order of each cell's atoms; a loop of one thread over all
// atoms for each took 546 us and 72 us for 5,000 atoms, 877 us and 118 us for 8,000 (one dependent
// load after another). Instead every atom is linked into a list of its binning cell and every N and O into
// one of a hashed 2 A cell (no extent of the receptor is needed); a carbon then looks at 27 buckets,
// most of them empty, and an atom ranks itself among the one or two of its cell: 5 + 7 + 6 us for
// 5,000 atoms, 5 + 9 + 6 us for 8,000 (cold caches), bound by the latency of a few dependent loads.

// Bucket of a 2 A cell (the multipliers of Teschner et al., "Optimized Spatial Hashing for Collision
// Detection of Deformable Objects", VMV 2003).
__device__ __forceinline__ unsigned polar_bucket(int x, int y, int z, unsigned mask) {
    return (((unsigned)x * 73856093u) ^ ((unsigned)y * 19349663u) ^ ((unsigned)z * 83492791u)) & mask;
}

// Links atom i into its cell's list: head[c] = 1 + the cell's last linked atom (0: none), next[i]
// likewise; and an N or O into the list of its 2 A cell's bucket.
__global__ void __launch_bounds__(128) receptor_link_kernel(const float* __restrict__ xyz, const uint8_t* __restrict__ el,
                                                            int n, CellGrid G, unsigned mask, int* __restrict__ cell_of,
                                                            int* __restrict__ head, int* __restrict__ next,
                                                            int* __restrict__ polar_head, int* __restrict__ polar_next,
                                                            int* __restrict__ cursor) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i == 0) *cursor = 0;
    const float x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
    const int e = el[i], c = cell_index(make_float4(x, y, z, 0.f), G.lo, G.inv_cell, G.cd);
    cell_of[i] = c;
    if (c >= 0) next[i] = atomicExch(head + c, i + 1);
    if (e == 1 || e == 2)
        polar_next[i] = atomicExch(polar_head + polar_bucket(__float2int_rd(0.5f * x), __float2int_rd(0.5f * y),
                                                             __float2int_rd(0.5f * z), mask), i + 1);
}

// XS type of each receptor atom: carbon is polar (C_P) iff an N or O lies within 1.75 A. A carbon's
// 27 buckets go to a group of lanes: kTypeLanes of them, each a few buckets.
constexpr int kTypeLanes = 8;
__device__ __forceinline__ void type_atom(const float* __restrict__ xyz, const uint8_t* __restrict__ el,
                                          const uint8_t* __restrict__ don, const uint8_t* __restrict__ acc, int n,
                                          unsigned mask, const int* __restrict__ polar_head,
                                          const int* __restrict__ polar_next, float4* __restrict__ typed, int slot) {
    const int i = slot / kTypeLanes, sub = slot % kTypeLanes;
    const bool live = i < n;
    float x = 0.f, y = 0.f, z = 0.f;
    int e = -1;
    if (live) {
        x = xyz[3 * i]; y = xyz[3 * i + 1]; z = xyz[3 * i + 2];
        e = el[i];
    }
    bool polar = false;
    if (e == 0) {
        const int cx = __float2int_rd(0.5f * x), cy = __float2int_rd(0.5f * y), cz = __float2int_rd(0.5f * z);
        int at[(27 + kTypeLanes - 1) / kTypeLanes];
#pragma unroll
        for (int m = 0; m < (27 + kTypeLanes - 1) / kTypeLanes; ++m) {
            const int k = sub + kTypeLanes * m;
            at[m] = k < 27 ? polar_head[polar_bucket(cx + k % 3 - 1, cy + (k / 3) % 3 - 1, cz + k / 9 - 1, mask)] : 0;
        }
#pragma unroll
        for (int m = 0; m < (27 + kTypeLanes - 1) / kTypeLanes; ++m)
            for (int a = at[m]; a && !polar; a = polar_next[a - 1]) {
                const int j = a - 1;
                const float dx = x - xyz[3 * j], dy = y - xyz[3 * j + 1], dz = z - xyz[3 * j + 2];
                polar = dx * dx + dy * dy + dz * dz < 1.75f * 1.75f;
            }
    }
    const unsigned near = __ballot_sync(PV_FULL, polar) >> ((threadIdx.x & 31) & ~(kTypeLanes - 1));
    if (live && sub == 0)
        typed[i] = make_float4(x, y, z, __int_as_float(xs_of(e, don[i], acc[i], near & ((1u << kTypeLanes) - 1u))));
}

// First atom of every cell: a warp per row of cells along x counts the row's cells (their lists hold
// one or two atoms each at a receptor's density), takes a run of the sorted atoms for the row from
// the cursor and writes the prefix. Rows land in any order; within a row cells are consecutive, and
// start[c + 1] ends cell c for every cell but a row's last (which lies beyond every box's reach).
__device__ __forceinline__ void start_row(const int* __restrict__ head, const int* __restrict__ next, const CellGrid& G,
                                          int* __restrict__ cursor, int* __restrict__ start, int row) {
    const int lane = threadIdx.x & 31;
    if (row >= G.cd[1] * G.cd[2]) return;
    const int c0 = row * G.cd[0];
    for (int pass = 0, base = 0; pass < 2; ++pass) {
        int run = base;
        for (int x0 = 0; x0 < G.cd[0]; x0 += 32) {
            const int x = x0 + lane;
            int k = 0;
            if (x < G.cd[0])
                for (int a = head[c0 + x]; a; a = next[a - 1]) ++k;
            int v = k;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(PV_FULL, v, o);
                if (lane >= o) v += u;
            }
            if (pass == 1 && x < G.cd[0]) start[c0 + x] = run + v - k;
            run += __shfl_sync(PV_FULL, v, 31);
            if (pass == 0 && G.cd[0] <= 32) {             // the usual row: one chunk, counted once
                int b = 0;
                if (lane == 0 && run) b = atomicAdd(cursor, run);
                b = __shfl_sync(PV_FULL, b, 0);
                if (x < G.cd[0]) start[c0 + x] = b + v - k;
                return;
            }
        }
        if (pass == 0) {
            if (lane == 0 && run) base = atomicAdd(cursor, run);
            base = __shfl_sync(PV_FULL, base, 0);
        }
    }
}

// Types and row starts, which do not depend on one another: the first type_blocks blocks type atoms.
__global__ void __launch_bounds__(128) receptor_type_kernel(
    const float* __restrict__ xyz, const uint8_t* __restrict__ el, const uint8_t* __restrict__ don,
    const uint8_t* __restrict__ acc, int n, CellGrid G, unsigned mask, const int* __restrict__ polar_head,
    const int* __restrict__ polar_next, float4* __restrict__ typed, const int* __restrict__ head,
    const int* __restrict__ next, int* __restrict__ cursor, int* __restrict__ start, int type_blocks) {
    if ((int)blockIdx.x < type_blocks)
        type_atom(xyz, el, don, acc, n, mask, polar_head, polar_next, typed, blockIdx.x * 128 + threadIdx.x);
    else
        start_row(head, next, G, cursor, start, ((int)blockIdx.x - type_blocks) * 4 + (threadIdx.x >> 5));
}

// Every atom to its place: its cell's first slot plus the number of the cell's atoms of lower index.
__global__ void __launch_bounds__(128) cell_scatter_kernel(const float4* __restrict__ typed,
                                                           const int* __restrict__ cell_of,
                                                           const int* __restrict__ head, const int* __restrict__ next,
                                                           const int* __restrict__ start, int n,
                                                           float4* __restrict__ sorted) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = cell_of[i];
    if (c < 0) return;
    int rank = 0;
    for (int a = head[c]; a; a = next[a - 1]) rank += a - 1 < i;
    sorted[start[c] + rank] = typed[i];
}

cudaError_t launch_receptor_prep(const float* xyz, const uint8_t* el, const uint8_t* don, const uint8_t* acc, int n,
                                 const float lo[3], float cell, const int cdims[3], float4* typed, int* cell_of,
                                 int* next, int* head, int* cell_start, float4* sorted, cudaStream_t s) {
    CellGrid G;
    for (int k = 0; k < 3; ++k) { G.lo[k] = lo[k]; G.cd[k] = cdims[k]; }
    G.inv_cell = 1.0f / cell;
    const int n_cells = cdims[0] * cdims[1] * cdims[2];
    // the N and O lists live in `sorted` (16 bytes per atom), which the last kernel alone writes: at
    // most 2 n bucket heads, then n links
    int buckets = 1;
    while (buckets < n) buckets <<= 1;
    int* polar_head = reinterpret_cast<int*>(sorted);
    int* polar_next = polar_head + buckets;
    // cleared together when one follows the other (but for padding)
    const ptrdiff_t gap = reinterpret_cast<char*>(polar_head) - reinterpret_cast<char*>(head + n_cells);
    const bool joined = gap >= 0 && gap <= 256;
    cudaError_t e = cudaMemsetAsync(head, 0, sizeof(int) * n_cells + (joined ? gap + sizeof(int) * buckets : 0), s);
    if (e == cudaSuccess && !joined) e = cudaMemsetAsync(polar_head, 0, sizeof(int) * buckets, s);
    if (e != cudaSuccess) return e;
    int* cursor = cell_start + n_cells;
    receptor_link_kernel<<<(n + 127) / 128, 128, 0, s>>>(xyz, el, n, G, (unsigned)buckets - 1u, cell_of, head, next,
                                                         polar_head, polar_next, cursor);
    const int type_blocks = (int)(((long long)n * kTypeLanes + 127) / 128);
    receptor_type_kernel<<<type_blocks + (cdims[1] * cdims[2] + 3) / 4, 128, 0, s>>>(
        xyz, el, don, acc, n, G, (unsigned)buckets - 1u, polar_head, polar_next, typed, head, next, cursor, cell_start,
        type_blocks);
    cell_scatter_kernel<<<(n + 127) / 128, 128, 0, s>>>(typed, cell_of, head, next, cell_start, n, sorted);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Map build
// ------------------------------------------------------------------------------------------
struct GridArgs {
    const float4* sorted;
    const int* cell_start;
    CellGrid G;
    const PvPocket* pockets;
    uint64_t slots_lo, slots_hi;
    int type_mask;
};

__device__ __forceinline__ int slot_from(uint64_t lo, uint64_t hi, int t) {
    uint64_t w = t < 8 ? lo : hi;
    return (int)(int8_t)((w >> (8 * (t < 8 ? t : t - 8))) & 0xff);
}

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

// Element classes of the ligand types in order of falling radius: S 2.0, C 1.9, N 1.8, O 1.7 A.
constexpr float class_radius(int k) { return k == 0 ? 2.0f : (k == 1 ? 1.9f : (k == 2 ? 1.8f : 1.7f)); }

// Surface distance from which the first Gaussian's term is under 2^-26 of the second's (3.75 d^2 +
// 1.5 d > 22.2 from ln of the two terms' ratio: d > 2.24), so that adding it leaves the sum as it is.
constexpr float kGauss1Reach = 2.3f;
constexpr int class_of(int t) { return t <= 1 ? 1 : (t <= 5 ? 2 : (t <= 9 ? 3 : 0)); }
__device__ __forceinline__ float hbond_ramp(float d) {
    return d < kHBondGood ? 1.0f : (d < kHBondBad ? -d * (1.0f / 0.7f) : 0.0f);
}

__device__ __forceinline__ float2 plus_term(float2 v, float w, float x, float y) {
    return make_float2(__fadd_rn(v.x, __fmul_rn(w, x)), __fadd_rn(v.y, __fmul_rn(w, y)));
}

// Maps of a tile of 8 x 8 x 4 nodes per CTA: a warp owns a block of 4 x 4 x 4 nodes, a lane two of them
// (z and z + 2), whose arithmetic is packed (FP32x2). CLASSES: the element classes asked for (bit k).
// Every node's sums run over the receptor atoms by cell, then input order.
//
// Bound by issue slots and the special-function unit: per (node, receptor atom within 8 A) a square
// root and two exponentials per element class. What keeps the rest down: the CTA stages only atoms
// within the cutoff of its tile's box, and a warp walks only those within the cutoff of its own block
// (1.1 A wide: three in four of the pairs it works on lie within the cutoff, against one in seven when
// every node met every atom of the neighbouring cells, the lanes of a warp spread over 2.6 x 1.1 A);
// repulsion, the hydrophobic ramp and hydrogen bonds run only where a lane is in their reach (a warp
// vote), and so does the first Gaussian, which farther out is too small to change the sum.
// Ten 24 A boxes of 8 types over 5,000 atoms: 1,312 -> 527 us, 4.7e8 warp instructions at 72 % of the
// issue peak; one 20 A box of 6 types over 2,000 atoms: 121 -> 54 us (4.5 CTAs per SM: a few warps
// per scheduler, each a serial walk). Tiles of 8 x 8 x 8 with 8 warps, whose waits at the staging
// barriers weigh more: 580 and 57 us. 7 CTAs per SM hold the registers at 72.
template <int CLASSES>
__global__ void __launch_bounds__(kGridThreads, 7) grid_kernel(GridArgs A) {
    __shared__ float4 s_atom[kStageCap];                 // xyz and XS radius of the atoms in reach
    __shared__ uint8_t s_flag[kStageCap];                // 1 hydrophobic, 2 donor, 4 acceptor
    __shared__ int s_row_start[kMaxRows * kMaxRows], s_row_off[kMaxRows * kMaxRows + 1];
    __shared__ int s_warp_n[kGridThreads / 32];
    __shared__ PvPocket P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < (int)(sizeof(PvPocket) / 4))
        reinterpret_cast<int*>(&P)[threadIdx.x] = reinterpret_cast<const int*>(A.pockets + blockIdx.y)[threadIdx.x];
    __syncthreads();
    const int tiles_x = (P.dims[0] + kTile - 1) / kTile, tiles_y = (P.dims[1] + kTile - 1) / kTile;
    const int tz = blockIdx.x / (tiles_x * tiles_y);
    if (tz * kTileZ >= P.dims[2]) return;                 // a pocket with fewer tiles than the largest
    const int t0[3] = {((int)blockIdx.x % tiles_x) * kTile, (((int)blockIdx.x / tiles_x) % tiles_y) * kTile, tz * kTileZ};
    // this warp's block of nodes and the lane's two nodes
    const int b0[3] = {t0[0] + 4 * (warp & 1), t0[1] + 4 * ((warp >> 1) & 1), t0[2] + 4 * (warp >> 2)};
    const bool warp_live = b0[0] < P.dims[0] && b0[1] < P.dims[1] && b0[2] < P.dims[2];
    const int ix = b0[0] + (lane & 3), iy = b0[1] + ((lane >> 2) & 3), iz0 = b0[2] + (lane >> 4), iz1 = iz0 + 2;
    const float px = P.origin[0] + ix * P.spacing, py = P.origin[1] + iy * P.spacing;
    const float2 pz = make_float2(P.origin[2] + iz0 * P.spacing, P.origin[2] + iz1 * P.spacing);
    // boxes of the tile's and of the warp's nodes, widened a little against the rounding of positions
    float tlo[3], thi[3], wlo[3], whi[3];
    float row_slack = 0.f;
    int c0[3], c1[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float far = fmaxf(fabsf(P.origin[k]), fabsf(P.origin[k] + P.dims[k] * P.spacing));
        const float slack = fminf(1e-4f + 1e-6f * far, 0.5f);
        row_slack = fmaxf(row_slack, 1e-2f + 2.f * slack);
        tlo[k] = P.origin[k] + t0[k] * P.spacing - slack;
        thi[k] = P.origin[k] + min(t0[k] + (k == 2 ? kTileZ : kTile), P.dims[k]) * P.spacing - P.spacing + slack;
        wlo[k] = P.origin[k] + b0[k] * P.spacing - slack;
        whi[k] = P.origin[k] + min(b0[k] + 4, P.dims[k]) * P.spacing - P.spacing + slack;
        c0[k] = max(0, (int)floorf((tlo[k] - kCutoff - A.G.lo[k]) * A.G.inv_cell));
        c1[k] = min(min(A.G.cd[k] - 2, c0[k] + kMaxRows - 1), (int)floorf((thi[k] + kCutoff - A.G.lo[k]) * A.G.inv_cell));
    }
    // the rows of cells in reach (each row's x range trimmed to the tile's box swept by the cutoff),
    // with the positions of their atoms in the row-concatenated list; warp 0 forms the prefix
    const int nrow_y = max(0, c1[1] - c0[1] + 1), nrow_z = max(0, c1[2] - c0[2] + 1);
    const int n_rows = (c1[0] >= c0[0]) ? nrow_y * nrow_z : 0;   // a tile is at most 7 x 4 A wide: 17 cells per axis
    const float cell = 1.0f / A.G.inv_cell;
    for (int r = threadIdx.x; r < n_rows; r += kGridThreads) {
        const int cy = c0[1] + r % nrow_y, cz = c0[2] + r / nrow_y;
        const float ylo = A.G.lo[1] + cy * cell, zlo = A.G.lo[2] + cz * cell;
        const float dy = fmaxf(0.f, fmaxf(ylo - thi[1], tlo[1] - (ylo + cell)) - row_slack);
        const float dz = fmaxf(0.f, fmaxf(zlo - thi[2], tlo[2] - (zlo + cell)) - row_slack);
        const float left = kCutoff2 - dy * dy - dz * dz;
        int b = 0, len = 0;
        if (left > 0.f) {
            const float half = sqrtf(left) + row_slack;
            const int x0 = max(c0[0], (int)floorf((tlo[0] - half - A.G.lo[0]) * A.G.inv_cell));
            const int x1 = min(c1[0], (int)floorf((thi[0] + half - A.G.lo[0]) * A.G.inv_cell));
            const int row = (cz * A.G.cd[1] + cy) * A.G.cd[0];
            if (x1 >= x0) {
                b = A.cell_start[row + x0];
                len = A.cell_start[row + x1 + 1] - b;
            }
        }
        s_row_start[r] = b;
        s_row_off[r + 1] = len;
    }
    __syncthreads();
    if (warp == 0) {
        int carry = 0;
        for (int r0 = 0; r0 < n_rows; r0 += 32) {
            int v = r0 + lane < n_rows ? s_row_off[r0 + lane + 1] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(PV_FULL, v, o);
                if (lane >= o) v += u;
            }
            if (r0 + lane < n_rows) s_row_off[r0 + lane + 1] = carry + v;
            carry += __shfl_sync(PV_FULL, v, 31);
        }
        if (lane == 0) s_row_off[0] = 0;
    }
    __syncthreads();
    const int total = s_row_off[n_rows];
    constexpr int kBase = (CLASSES & 1) ? 0 : (CLASSES & 2) ? 1 : (CLASSES & 4) ? 2 : 3;   // widest class
    float2 sum[PV_N_XS];
#pragma unroll
    for (int t = 0; t < PV_N_XS; ++t) sum[t] = splat(0.f);

    int staged = 0;
    for (int base = 0; base < total; base += kGridThreads) {
        // stage, in list order, the atoms within the cutoff of the tile's box
        const int g = base + threadIdx.x;
        bool take = false;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g < total) {
            int lo_r = 0, hi_r = n_rows - 1;             // the last row whose atoms begin at or before g
            while (lo_r < hi_r) {
                const int mid = (lo_r + hi_r + 1) >> 1;
                if (s_row_off[mid] <= g) lo_r = mid; else hi_r = mid - 1;
            }
            a = A.sorted[s_row_start[lo_r] + (g - s_row_off[lo_r])];
            const float ex = fmaxf(0.f, fmaxf(tlo[0] - a.x, a.x - thi[0])), ey = fmaxf(0.f, fmaxf(tlo[1] - a.y, a.y - thi[1])),
                        ez = fmaxf(0.f, fmaxf(tlo[2] - a.z, a.z - thi[2]));
            take = ex * ex + ey * ey + ez * ez < kCutoff2;
        }
        const unsigned bal = __ballot_sync(PV_FULL, take);
        if (lane == 0) s_warp_n[warp] = __popc(bal);
        __syncthreads();
        int at = staged + __popc(bal & ((1u << lane) - 1u)), add = 0;
#pragma unroll
        for (int w = 0; w < kGridThreads / 32; ++w) {
            const int v = s_warp_n[w];
            at += w < warp ? v : 0;
            add += v;
        }
        if (take) {
            const int tj = __float_as_int(a.w);
            s_atom[at] = make_float4(a.x, a.y, a.z, xs_radius(tj));
            s_flag[at] = (uint8_t)((xs_hydrophobic(tj) ? 1 : 0) | (xs_donor(tj) ? 2 : 0) | (xs_acceptor(tj) ? 4 : 0));
        }
        staged += add;
        __syncthreads();
        if (base + kGridThreads < total && staged + kGridThreads <= kStageCap) continue;
        // the staged atoms, 32 at a time: those within the cutoff of the warp's block, in order
        for (int k0 = 0; warp_live && k0 < staged; k0 += 32) {
            bool near = false;
            if (k0 + lane < staged) {
                const float4 q = s_atom[k0 + lane];
                const float ex = fmaxf(0.f, fmaxf(wlo[0] - q.x, q.x - whi[0])), ey = fmaxf(0.f, fmaxf(wlo[1] - q.y, q.y - whi[1])),
                            ez = fmaxf(0.f, fmaxf(wlo[2] - q.z, q.z - whi[2]));
                near = ex * ex + ey * ey + ez * ez < kCutoff2;
            }
            for (unsigned m = __ballot_sync(PV_FULL, near); m; m &= m - 1) {
                const int t = k0 + __ffs(m) - 1;
                const float4 q = s_atom[t];
                const float dx = px - q.x, dy = py - q.y;
                const float dxy = dx * dx + dy * dy;
                const float2 dz = __fadd2_rn(pz, splat(-q.z));
                float2 r2 = __ffma2_rn(dz, dz, splat(dxy));
                // beyond the cutoff: a distance at which every term below is zero
                r2.x = r2.x < kCutoff2 ? r2.x : 1e6f;
                r2.y = r2.y < kCutoff2 ? r2.y : 1e6f;
                const float2 r = make_float2(sqrtf(r2.x), sqrtf(r2.y));
                float2 d[4], v[4];                       // surface distance and the steric terms per class
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (!((CLASSES >> k) & 1)) continue;
                    d[k] = __fadd2_rn(__fadd2_rn(r, splat(-class_radius(k))), splat(-q.w));
                    const float2 b = __fadd2_rn(d[k], splat(-3.0f));
                    const float2 a2 = __fmul2_rn(__fmul2_rn(b, b), splat(-0.25f * kLog2e));
                    v[k] = __fmul2_rn(splat(kWGauss2), make_float2(exp2_approx(a2.x), exp2_approx(a2.y)));
                }
                const float d_min = fminf(d[kBase].x, d[kBase].y);
                if (__any_sync(PV_FULL, d_min < kGauss1Reach)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (!((CLASSES >> k) & 1)) continue;
                        const float2 a1 = __fmul2_rn(__fmul2_rn(d[k], d[k]), splat(-4.0f * kLog2e));
                        v[k] = __ffma2_rn(splat(kWGauss1), make_float2(exp2_approx(a1.x), exp2_approx(a1.y)), v[k]);
                    }
                }
                if (!__any_sync(PV_FULL, d_min < kHydBad)) {
#pragma unroll
                    for (int t = 0; t < PV_N_XS; ++t)
                        if ((CLASSES >> class_of(t)) & 1) sum[t] = __fadd2_rn(sum[t], v[class_of(t)]);
                    continue;
                }
                const int flag = s_flag[t];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (!((CLASSES >> k) & 1)) continue;
                    const float2 rep = make_float2(fminf(d[k].x, 0.f), fminf(d[k].y, 0.f));
                    v[k] = __ffma2_rn(__fmul2_rn(rep, splat(kWRepulsion)), rep, v[k]);
                    if (k == 0) sum[10] = __fadd2_rn(sum[10], v[k]);
                    if (k == 1) {
                        float2 vh = v[k];
                        if (flag & 1)
                            vh = plus_term(vh, kWHydrophobic, __saturatef(kHydBad - d[k].x), __saturatef(kHydBad - d[k].y));
                        sum[0] = __fadd2_rn(sum[0], vh);
                        sum[1] = __fadd2_rn(sum[1], v[k]);
                    }
                    if (k >= 2) {
                        // types without flags, donor, acceptor, both: a donor bonds with acceptors, ...
                        float2* s = sum + (k == 2 ? 2 : 6);
                        s[0] = __fadd2_rn(s[0], v[k]);
                        if (flag & 6) {
                            const float2 vb = plus_term(v[k], kWHBond, hbond_ramp(d[k].x), hbond_ramp(d[k].y));
                            s[1] = __fadd2_rn(s[1], (flag & 4) ? vb : v[k]);
                            s[2] = __fadd2_rn(s[2], (flag & 2) ? vb : v[k]);
                            s[3] = __fadd2_rn(s[3], vb);
                        } else {
                            s[1] = __fadd2_rn(s[1], v[k]);
                            s[2] = __fadd2_rn(s[2], v[k]);
                            s[3] = __fadd2_rn(s[3], v[k]);
                        }
                    }
                }
            }
        }
        if (base + kGridThreads >= total) break;
        staged = 0;
        __syncthreads();
    }
    if (ix >= P.dims[0] || iy >= P.dims[1]) return;
#pragma unroll
    for (int t = 0; t < PV_N_XS; ++t) {
        if (!((A.type_mask >> t) & 1)) continue;
        if (!((CLASSES >> class_of(t)) & 1)) continue;
        float* m = P.maps + (long long)slot_from(A.slots_lo, A.slots_hi, t) * P.nxyz + (iy * P.dims[0] + ix);
        if (iz0 < P.dims[2]) m[(long long)iz0 * P.nxy] = sum[t].x;
        if (iz1 < P.dims[2]) m[(long long)iz1 * P.nxy] = sum[t].y;
    }
}

// Cell-packed copies of pockets' maps: a thread takes a column of kPackZ cells of one map, whose
// upper corners become the next cell's lower ones, so a cell costs four loads (three of them
// L1 hits of its neighbours' lines) and one 32-byte store; a warp stores 1 KB without a gap. Bound by
// the stores: 671 MB written and 88 MB read for ten 24 A boxes of 8 types in 214 us as a launch per
// pocket of one cell per thread, its two 16-byte stores 32 bytes apart and its index divided out of a
// 64-bit cell number; 113 us for the one launch, 6.7 TB/s.
constexpr int kPackZ = 8;
__global__ void __launch_bounds__(128) pack_cells_kernel(const PvPocket* __restrict__ pockets, int n_chunks) {
    const PvPocket& P = pockets[blockIdx.z];
    const int cx = P.dims[0] - 1, cy = P.dims[1] - 1, cz = P.dims[2] - 1;
    const int slot = blockIdx.y / n_chunks, iz0 = (blockIdx.y - slot * n_chunks) * kPackZ;
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= cx * cy || iz0 >= cz) return;
    const int iy = col / cx, ix = col - iy * cx;
    const int nx = P.dims[0], nxy = P.nxy, n = min(kPackZ, cz - iz0);
    const float* m = P.maps + (long long)slot * P.nxyz + ((long long)iz0 * nxy + iy * nx + ix);
    float* out = reinterpret_cast<float*>(const_cast<float4*>(P.cells)) +
                 8 * ((long long)slot * P.ncells + (long long)iz0 * (cx * cy) + col);
    const bool wide = (reinterpret_cast<uintptr_t>(P.cells) & 31) == 0;   // a caller's allocator may align to 16 bytes
    float4 lo = make_float4(__ldg(m), __ldg(m + 1), __ldg(m + nx), __ldg(m + nx + 1));
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        m += nxy;
        const float4 hi = make_float4(__ldg(m), __ldg(m + 1), __ldg(m + nx), __ldg(m + nx + 1));
        if (wide) {
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out), "f"(lo.x), "f"(lo.y),
                         "f"(lo.z), "f"(lo.w), "f"(hi.x), "f"(hi.y), "f"(hi.z), "f"(hi.w)
                         : "memory");
        } else {
            reinterpret_cast<float4*>(out)[0] = lo;
            reinterpret_cast<float4*>(out)[1] = hi;
        }
        lo = hi;
        out += 8LL * cx * cy;
    }
}

cudaError_t launch_pack_cells(const PvPocket* pockets_dev, const PvPocket* pockets_host, int first, int n,
                              int n_maps, cudaStream_t s) {
    // blockIdx: columns of a map, (map slot, chunk of z), pocket
    auto extent = [&](int p) {
        const int* d = pockets_host[p].dims;
        return RunExtent{((d[0] - 1) * (d[1] - 1) + 127) / 128, (long long)((d[2] - 1 + kPackZ - 1) / kPackZ) * n_maps};
    };
    return launch_runs(first, n, extent, [&](int p0, int np, RunExtent most) {
        pack_cells_kernel<<<dim3((unsigned)most.x, (unsigned)most.y, np), 128, 0, s>>>(pockets_dev + p0, (int)most.y / n_maps);
        return cudaGetLastError();
    });
}

cudaError_t launch_grid_maps(const float4* sorted, const int* cell_start, const float lo[3], float cell,
                             const int cdims[3], const PvPocket* pockets_dev, const PvPocket* pockets_host, int n_pockets,
                             uint64_t slots_lo, uint64_t slots_hi, int type_mask, cudaStream_t s) {
    GridArgs a;
    a.sorted = sorted;
    a.cell_start = cell_start;
    for (int k = 0; k < 3; ++k) { a.G.lo[k] = lo[k]; a.G.cd[k] = cdims[k]; }
    a.G.inv_cell = 1.0f / cell;
    a.slots_lo = slots_lo;
    a.slots_hi = slots_hi;
    a.type_mask = type_mask;
    using Kernel = void (*)(GridArgs);
    static const Kernel kernels[16] = {nullptr,          grid_kernel<1>,  grid_kernel<2>,  grid_kernel<3>,
                                       grid_kernel<4>,   grid_kernel<5>,  grid_kernel<6>,  grid_kernel<7>,
                                       grid_kernel<8>,   grid_kernel<9>,  grid_kernel<10>, grid_kernel<11>,
                                       grid_kernel<12>,  grid_kernel<13>, grid_kernel<14>, grid_kernel<15>};
    const int classes = ((type_mask & 0x400) ? 1 : 0) | ((type_mask & 0x3) ? 2 : 0) | ((type_mask & 0x3c) ? 4 : 0) |
                        ((type_mask & 0x3c0) ? 8 : 0);
    if (!classes) return cudaErrorInvalidValue;
    // blockIdx.y is the pocket, blockIdx.x its tile
    auto extent = [&](int p) {
        const int* d = pockets_host[p].dims;
        return RunExtent{(long long)((d[0] + kTile - 1) / kTile) * ((d[1] + kTile - 1) / kTile) * ((d[2] + kTileZ - 1) / kTileZ), 1};
    };
    return launch_runs(0, n_pockets, extent, [&](int p0, int np, RunExtent most) {
        a.pockets = pockets_dev + p0;
        kernels[classes]<<<dim3((unsigned)most.x, np), kGridThreads, 0, s>>>(a);
        return cudaGetLastError();
    });
}

}  // namespace pv
