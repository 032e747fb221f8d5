#include "idkm_mma_loop_impl.cuh"
namespace idkm {
extern const MmaLoopEntry k_mma_loop_d2[N_MMA_LOOP] = IDKM_LOOP_ROW_2(false, IDKM_GRP(2, 16, 16, false));
}
