#include "idkm_mma_loop_impl.cuh"
namespace idkm {
extern const MmaLoopEntry k_mma_loop_d4[N_MMA_LOOP] = IDKM_LOOP_ROW_4(false);
}
