// eval_small.cu -- the field kernels for scenes without a BVH and without a
// candidate list (see CREEP_SMALL).
#define CREEP_SMALL
#include "eval_fields.cu"
