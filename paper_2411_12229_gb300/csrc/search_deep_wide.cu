// search_deep_wide.cu -- the deep-beam search kernel (search_deep.cuh) for
// 512 < d <= 2048 (CH = 8, 12, 16): 9 to 13 resident warps per SM, bounded by
// the vertex blocks and beams in shared memory, so every build may use many
// registers.
#include "search_deep.cuh"

namespace sqg {

#define SQG_DEEP_WIDE_SWITCH(CALL)              \
    switch (ch * 100 + nr * 10 + rk) {          \
        case 811: return CALL(8, 1, 1, 3);      \
        case 814: return CALL(8, 1, 4, 3);      \
        case 821: return CALL(8, 2, 1, 3);      \
        case 824: return CALL(8, 2, 4, 3);      \
        case 1211: return CALL(12, 1, 1, 3);    \
        case 1214: return CALL(12, 1, 4, 3);    \
        case 1221: return CALL(12, 2, 1, 3);    \
        case 1224: return CALL(12, 2, 4, 3);    \
        case 1611: return CALL(16, 1, 1, 3);    \
        case 1614: return CALL(16, 1, 4, 3);    \
        case 1621: return CALL(16, 2, 1, 2);    \
        case 1624: return CALL(16, 2, 4, 2);    \
        default: return cudaErrorInvalidValue;  \
    }

cudaError_t launch_search_deep_wide(int ch, int nr, int rk, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                    const SearchArgs &a) {
#define CALL(C, R, K, M) deep_launch_one<C, R, K, M>(grid, block, smem, s, a)
    SQG_DEEP_WIDE_SWITCH(CALL)
#undef CALL
}

cudaError_t search_occupancy_deep_wide(int ch, int nr, int rk, int block, size_t smem, int *blocks_per_sm) {
#define CALL(C, R, K, M) deep_occ_one<C, R, K, M>(block, smem, blocks_per_sm)
    SQG_DEEP_WIDE_SWITCH(CALL)
#undef CALL
}

}  // namespace sqg
