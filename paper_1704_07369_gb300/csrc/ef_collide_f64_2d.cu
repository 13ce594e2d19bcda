// FP64 collide kernel instantiations, 2D.
#define EF_D 2
#define EF_SUF f64_2d
#include "ef_collide_q_variant.inc"
