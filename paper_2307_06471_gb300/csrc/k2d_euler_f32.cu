// 2D kernels: PHYS_EULER in float
#define CRK_T float
#define CRK_PHYS crk::PHYS_EULER
#define CRK_NAME euler_f32
// square cells take the square-cell form of the step (k2d_euler_f32_sq.cu)
#define CRK_SQ_STEP 1
#include "kernels_2d.inc"
