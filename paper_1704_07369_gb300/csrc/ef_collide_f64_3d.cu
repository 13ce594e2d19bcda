// FP64 collide kernel instantiations, 3D.
#define EF_D 3
#define EF_SUF f64_3d
#include "ef_collide_q_variant.inc"
