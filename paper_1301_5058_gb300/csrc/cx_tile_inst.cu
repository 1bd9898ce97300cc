// cx_tile_inst.cu -- explicit instantiations of the register-tile pass
// (cx_tile_kernels.cuh).  The build compiles this file once per (precision,
// chemotaxis law, mobility), given as CX_INST_PREC (0 FP64: no kernels here,
// 1 FP32), CX_INST_LAW and CX_INST_MOB, so that the sets of kernels compile in
// parallel; without the macros it instantiates all of them.
#include "cx_tile_kernels.cuh"

namespace cx {
namespace tile {

#define CX_TILE_INST(LAW, MOB)                                                                 \
    template cudaError_t launch_tile_lm<LAW, MOB>(const TileLaunch &, const TilePlan &, bool,  \
                                                  cudaStream_t);

#if defined(CX_INST_PREC) && defined(CX_INST_LAW) && defined(CX_INST_MOB)
#if CX_INST_PREC == 1
CX_TILE_INST(CX_INST_LAW, CX_INST_MOB)
#endif
#else
CX_TILE_INST(CX_CHEMO_RECEPTOR, CX_MOBILITY_CENTRAL)
CX_TILE_INST(CX_CHEMO_RECEPTOR, CX_MOBILITY_UPWIND)
CX_TILE_INST(CX_CHEMO_CONSTANT, CX_MOBILITY_CENTRAL)
CX_TILE_INST(CX_CHEMO_CONSTANT, CX_MOBILITY_UPWIND)
#endif

}  // namespace tile
}  // namespace cx
