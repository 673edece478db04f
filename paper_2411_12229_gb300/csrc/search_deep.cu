// search_deep.cu -- the deep-beam search kernel (search_deep.cuh) for d <=
// 512, and the dispatch to the instantiations for larger d
// (search_deep_wide.cu).
#include "search_deep.cuh"

namespace sqg {

// (d chunks CH, neighbours per lane NR, result slots per lane RK) -> the
// instantiation and the resident blocks per SM it is built for
#define SQG_DEEP_SWITCH(CALL)                   \
    switch (ch * 100 + nr * 10 + rk) {          \
        case 111: return CALL(1, 1, 1, 8);      \
        case 114: return CALL(1, 1, 4, 7);      \
        case 121: return CALL(1, 2, 1, 6);      \
        case 124: return CALL(1, 2, 4, 6);      \
        case 211: return CALL(2, 1, 1, 7);      \
        case 214: return CALL(2, 1, 4, 6);      \
        case 221: return CALL(2, 2, 1, 6);      \
        case 224: return CALL(2, 2, 4, 5);      \
        case 411: return CALL(4, 1, 1, 4);      \
        case 414: return CALL(4, 1, 4, 4);      \
        case 421: return CALL(4, 2, 1, 4);      \
        case 424: return CALL(4, 2, 4, 4);      \
        default: return cudaErrorInvalidValue;  \
    }

cudaError_t launch_search_deep(int ch, int nr, int rk, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                               const SearchArgs &a) {
    if (ch > 4) return launch_search_deep_wide(ch, nr, rk, grid, block, smem, s, a);
#define CALL(C, R, K, M) deep_launch_one<C, R, K, M>(grid, block, smem, s, a)
    SQG_DEEP_SWITCH(CALL)
#undef CALL
}

cudaError_t search_occupancy_deep(int ch, int nr, int rk, int block, size_t smem, int *blocks_per_sm) {
    if (ch > 4) return search_occupancy_deep_wide(ch, nr, rk, block, smem, blocks_per_sm);
#define CALL(C, R, K, M) deep_occ_one<C, R, K, M>(block, smem, blocks_per_sm)
    SQG_DEEP_SWITCH(CALL)
#undef CALL
}

}  // namespace sqg
