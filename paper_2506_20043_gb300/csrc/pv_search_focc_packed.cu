// pv_search_focc_packed.cu -- the round kernels with the first-order consistency check (Eq. 4-5)
// reading cell-packed maps: the eight variants of pv_search_focc.cu for that layout.
#include "pv_chain.cuh"

namespace pv {

const void* search_focc_packed_kernel(int variant) {
    static const void* const kFns[kSearchVariants] = {
        (const void*)search_round_kernel<512, 32, true, 1>, (const void*)search_round_kernel<640, 32, true, 1>,
        (const void*)search_round_kernel<768, 32, true, 1>, (const void*)search_round_kernel<896, 32, true, 1>,
        (const void*)search_round_kernel<512, 16, true, 1>, (const void*)search_round_kernel<640, 16, true, 1>,
        (const void*)search_round_kernel<768, 16, true, 1>, (const void*)search_round_kernel<1024, 16, true, 1>,
    };
    if (variant == kSearchFew) return (const void*)search_few_kernel<true, 1>;
    return variant >= 0 && variant < kSearchVariants ? kFns[variant] : nullptr;
}

}  // namespace pv
