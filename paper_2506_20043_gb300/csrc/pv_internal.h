// pv_internal.h -- kernel launchers shared between the runtime (pv_api.cu) and the kernels.
#pragma once
#include <stdint.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include "pv_layout.h"

struct pv_context;

namespace pv {

// A named NVTX range over a host scope: a profiler's timeline shows each library call and, inside a
// dock, its autotuning, search rounds and selection (ranges cost a few nanoseconds without a tool).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// Context access for entry points defined outside pv_api.cu (false on a bad handle).
bool context_device_stream(pv_context* ctx, int* device, cudaStream_t* stream);
void context_set_error(pv_context* ctx, const char* msg);
// Whether any of the host arrays is page-locked (cudaMallocHost or registered): copies from them
// run asynchronously, so a call that must not retain them waits for those copies.
bool host_pinned(const void* a, const void* b, const void* c, const void* d);

constexpr int kSearchThreadsMax = 512;
constexpr int kTopkThreads = 256;
constexpr int kMaxTopK = 32;
constexpr int kMaxMergeEntries = 8192;

// ---- grid cache (pv_grid.cu) ----
// XS typing of receptor atoms, typed[i] = (x, y, z, type as int bits), and their binning into cubic
// cells of edge `cell` over the region lo + [0, cdims * cell): sorted holds them by cell, in input order
// within a cell, cells consecutive along x (cell_start[c] .. cell_start[c + 1] for every cell but the
// last of a row); atoms outside the region are typed but not binned. cell_of, next: [n], head: [cells],
// cell_start: [cells + 1].
cudaError_t launch_receptor_prep(const float* xyz, const uint8_t* el, const uint8_t* don, const uint8_t* acc, int n,
                                 const float lo[3], float cell, const int cdims[3], float4* typed, int* cell_of,
                                 int* next, int* head, int* cell_start, float4* sorted, cudaStream_t s);
// Map build of n_pockets pockets (their device records and the same records on the host).
cudaError_t launch_grid_maps(const float4* sorted, const int* cell_start, const float lo[3], float cell,
                             const int cdims[3], const PvPocket* pockets_dev, const PvPocket* pockets_host, int n_pockets,
                             uint64_t slots_lo, uint64_t slots_hi, int type_mask, cudaStream_t s);

// Cell-packed copies of the maps of pockets [first, first + n) of a device pocket table: for every
// map slot and cell, its eight corner values as two float4 at P.cells.
cudaError_t launch_pack_cells(const PvPocket* pockets_dev, const PvPocket* pockets_host, int first, int n,
                              int n_maps, cudaStream_t s);

// ---- scoring (pv_score.cu) ----
// pocket: device pointer to the pocket record (its maps pointers included); layout: the maps read,
// 0 plain, 1 cell-packed (the pocket must hold them)
cudaError_t launch_score(const PvLigBlob* lig, int lig_bytes, const PvPocket* pocket,
                         PvSlots slots, int n_poses, int pot_stride,
                         const float* pose, float* energy, float* grad, float* parts,
                         const float* grad_energy, float* grad_pose, float* grad_xyz,
                         int layout, cudaStream_t s);
// SF of posed atom coordinates [n][n_atoms][3] (input order); energy and grad_xyz nullable,
// grad_xyz scaled by grad_energy (nullable: 1).
cudaError_t launch_score_xyz(const PvLigBlob* lig, int lig_bytes, const PvPocket* pocket, PvSlots slots,
                             int n_poses, const float* xyz, const float* grad_energy, float* energy,
                             float* grad_xyz, int layout, cudaStream_t s);
cudaError_t launch_pose_coords(const PvLigBlob* lig, int lig_bytes, int n_poses, int pot_stride,
                               const float* pose, float* xyz, cudaStream_t s);

// ---- gather microbenchmark (pv_probe.cu) ----
// n_points trilinear interpolations (value + gradient) at hashed positions in the box of a hashed
// pocket of the device table, on hashed map slots in [0, n_slots); sink is written only in a case
// that does not occur.
cudaError_t launch_gather_probe(const PvPocket* pockets_dev, int n_pockets, int n_slots, long long n_points,
                                uint32_t seed, float* sink, int n_sm, int layout, cudaStream_t s);

// ---- search (pv_search.cu) ----
struct SearchArgs {
    const int* order;              // pairs in the order they are worked on
    int n_items;                   // step blocks x items_per_block
    int* queue;                    // work counter of this round (zeroed before the launch)
    int items_per_pair;            // batched: an item is item_units warp loads of chains of one pair
    int item_units;                //          (a warp load: one chain, or two on half warps)
    int units;                     // batched: warp loads per pair
    int lig_slots;                 // batched: ligand records a CTA stages at a time, 1 .. kLigSlots
    const PvPairDesc* pairs;
    const PvLigBlob* const* ligs;  // device pointer table
    const PvPocket* pockets;
    uint64_t slots_lo, slots_hi;   // XS type -> map slot, 8 bits per type
    float* chains;                 // [n_pairs * chains][PV_CHAIN_STRIDE]
    float* ring;                   // [n_pairs * chains][PV_RING_STRIDE] when C.focc > 0, else null
    PvSearchConst C;
    int step0, step1;              // the launch's MC steps
    int items_per_block;           // batched: work items of one step block
    int block_steps;               // batched: MC steps per block; block b covers step0 + b * block_steps ..
    int* progress;                 // batched: step blocks finished per warp load of chains
    int lig_smem_bytes;            // staging capacity for one ligand
    const unsigned long long* t0;  // start time of the dock (globaltimer)
    unsigned long long timeout_ns; // 0 = none
    unsigned long long wait_ns;    // batched: bound on a step block's wait for its predecessor, and on a warp's for a
                                   // ligand slot
    int* err;
    unsigned long long* evals;
    int layout;                    // map layout the kernel reads: 0 plain, 1 cell-packed
};
constexpr int kLigSlots = 4;
// MC steps of a step block, of the `steps` of a launch. When every unit of work runs at once there is nothing to hand
// over, and a warp keeps its chains to the end (blocks would make the fast chains wait for the slow ones'
// hand-outs); else blocks of about 1/32 of the steps, so that the last ones spread over the SMs. A caller who fixes
// the CTA size gets blocks of about 1/16 (at least 25 steps). No block that is handed over is longer than
// kMaxBlockSteps (a second of a large ligand's chain on a full GPU): warps that wait for a chain's block, or for
// a ligand slot that its warp holds, would wait as long. Longer again where the items would not fit an int.
constexpr int kMaxBlockSteps = 512;
inline int step_block(int steps, bool fixed_cta, bool all_resident, int items_per_block) {
    if (all_resident && !fixed_cta) return steps;
    const int part = fixed_cta ? (steps > 400 ? (steps - 1) / 16 + 1 : 25) : (steps > 256 ? (steps - 1) / 32 + 1 : 8);
    const long long least = ((long long)steps * items_per_block >> 30) + 1;
    const int block = part < kMaxBlockSteps ? part : kMaxBlockSteps;
    return least > block ? (int)least : block;
}
int search_smem_bytes(int lig_bytes, int warps, int lanes, int lig_slots);
// Variants of the round kernel: 0-3 run a chain per warp, 4-7 a chain per half warp (ligands of
// at most 32 atoms and 10 torsions); within each group the launch bounds are 512, 640, 768 and 896
// (half warps: 1,024) threads per SM, i.e. decreasing register budgets.
constexpr int kSearchVariants = 8;
int search_variant_max_warps(int variant);     // the warps_per_cta a caller may ask for
int search_variant_sm_warps(int variant);      // warps per SM the register budget is for
int search_variant_lanes(int variant);
cudaError_t search_max_ctas_per_sm(int variant, bool focc, int layout, int warps, int smem, int* out);
// The round kernel of a variant with the consistency check (Eq. 4-5) compiled in (pv_search_focc.cu),
// and the variants reading cell-packed maps without and with the check (pv_search_packed.cu,
// pv_search_focc_packed.cu).
const void* search_focc_kernel(int variant);
const void* search_packed_kernel(int variant);
const void* search_focc_packed_kernel(int variant);
constexpr int kSearchFew = kSearchVariants;    // index of the kernel for few chains beside the variants
constexpr int kFewWarps = 8;                   // warps of one chain there
bool search_few_fits(bool focc, int layout, int lig_bytes, int n, int sms);
cudaError_t launch_search_few(const SearchArgs& a, int n, cudaStream_t s);
cudaError_t launch_search_round(const SearchArgs& a, int variant, int grid, int warps, cudaStream_t s);
constexpr int kPlainWarps = 4;                 // warps per CTA of the thread-per-chain form
cudaError_t launch_plain_search(const SearchArgs& a, int pair, const PvLigBlob* lig_dev,
                                cudaStream_t s);
cudaError_t launch_mark_t0(unsigned long long* t0, cudaStream_t s);

struct TopkArgs {
    const PvPairDesc* pairs;
    const PvLigBlob* const* ligs;
    const PvPocket* pockets;
    uint64_t slots_lo, slots_hi;
    const float* chains;
    PvSearchConst C;
    int lig_smem_bytes;
    PvPoseRec* poses;              // [n_pairs][top_k]
    float* pots;                   // [n_pairs][top_k][pot_stride]
    float* xyz;                    // [n_pairs][top_k][atom_stride][3]
    int* n_kept;                   // [n_pairs]
    int* status;                   // [n_pairs]
    int pair0;                     // first pair handled by this launch
};
cudaError_t prepare_topk(const TopkArgs& a);   // raise shared-memory limits before capture
cudaError_t launch_topk(const TopkArgs& a, int n_pairs, cudaStream_t s);

struct MergeArgs {
    const int* lig_pair_start;     // [n_ligs + 1] CSR of pairs per ligand
    const int* lig_pairs;          // pair ids
    const PvPoseRec* poses;
    const int* n_kept;
    int top_k;
    int rank_stride;
    int* ranking;                  // [n_ligs][rank_stride]
};
cudaError_t prepare_merge(int max_entries);
cudaError_t launch_merge(const MergeArgs& a, int n_ligs, int max_entries, cudaStream_t s);

}  // namespace pv
