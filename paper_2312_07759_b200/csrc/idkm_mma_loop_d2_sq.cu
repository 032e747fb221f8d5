#include "idkm_mma_loop_impl.cuh"
namespace idkm {
// (squared distance, k > 128: a launch per iteration is as fast: 15.6 against 17.3 us at 4 K pairs, 155 against 160 at 1 M)
#define IDKM_GRP_NONE { nullptr, 256, 0 }
extern const MmaLoopEntry k_mma_loop_d2_sq[N_MMA_LOOP] = IDKM_LOOP_ROW_2(true, IDKM_GRP_NONE);
}
