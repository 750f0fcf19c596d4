// Batched Dslash, spinor storage F32, links read past L1 (stream_links in launch.h). A
// translation unit of its own, compiled in parallel with kernels_f32.cu.
#define LQCD_SP lqcd::P_F32
#define LQCD_SFX f32
#define LQCD_STREAM_UNIT 1
#include "kernels_inst.cuh"
